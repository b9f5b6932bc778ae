// Parallel QR of banded matrices (Sec. 4.4) by row compression and block cyclic reduction.
//
// An instance has N columns, cut into G = ceil(N / 8) blocks of 8 (the last block padded
// with "virtual" columns that carry a unit damping row and nothing else, so that the padded
// matrix has full rank and the real columns' solution is unchanged).  Every row has at most
// 8 consecutive entries, so a row whose first column lies in block g touches blocks g and
// g + 1 only.
//
//   1. compress   per block g, the Householder QR (Sec. 2) of all rows starting in block g
//                 plus the damping rows lambda^(1/2) D_j of the block's columns (the row
//                 interleave of Sec. 4.5 / 5.2) reduces them to a 16 x 16 upper-trapezoidal
//                 block row E_g = [A_g | B_g] on blocks (g, g + 1).  Row-heavy groups are split
//                 over several threads whose partial triangles are merged.
//   2. reduce     level l works on the block rows F_i of blocks b_i = i 2^l: for every odd
//                 i, QR of [F_{i-1}; F_i] with block b_i's columns first gives the 8 rows of R
//                 for b_i (coupled to b_{i-1} and b_{i+1}) and a new 16-row block row on
//                 (b_{i-1}, b_{i+1}); an unpaired last block row moves up unchanged; at one
//                 block row the last R rows come out.  All eliminations of a level run in
//                 parallel, ceil(log2 G) + 1 levels.
//   3. solve      back-substitution level by level from the top: R_bb x_b = c_b - R_left
//                 x_{b - 2^l} - R_right x_{b + 2^l} for all blocks of a level in parallel.
// The product is a QR factorization of the matrix with its columns in nested-dissection
// order (the blocks of the lowest level first), so R differs from the natural-order banded
// R; R^T R = A^T A and the solution are the same.  Refinement solves R^T h = g level by level
// upwards, then R dx = h.  An instance's upper levels (at most kTailBlocks blocks left) run in one
// CTA, levels and back-substitution together: their launches cost more than their work.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <string>
#include <vector>

#include "chain.cuh"
#include "device_util.cuh"
#include "f32x2.cuh"
#include "internal.h"
#include "roots.cuh"
#include "sums.cuh"

namespace qrkit {
namespace {

constexpr int kCB = 8;              // columns per block
constexpr int kE0 = 144;            // compressed block row: 8 rows x 8 | 8 rows x 8 | rhs 16 (below)
constexpr int kFW = 208;            // block row: A 8 x 8 | B 16 x 8 | rhs 16
constexpr int kRW = 200;            // R block row: own 8 x 8 | left 8 x 8 | right 8 x 8 | rhs 8
constexpr int64_t kTailBlocks = 128;

__device__ __forceinline__ void cr_record(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// Square root and reciprocal of the fronts' reflectors: the hardware approximations for float
// (sqrt.approx / rcp.approx, about one ulp; a row meets few of these reflectors), IEEE for double.
__device__ __forceinline__ float qr_sqrt(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double qr_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float qr_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double qr_rcp(double x) { return 1.0 / x; }

// Squared norms of float columns below 2^-90 lose bits, and vanish below 2^-149: the column is then squared again times
// kLift.  (A reflector of few rows meets pivots far below the scale of the data.)
constexpr float kLift = 0x1p80f;
template <typename T>
__device__ __forceinline__ bool faint(T n2) {
  return sizeof(T) == 4 && n2 < T(0x1p-90f);
}

// The Householder reflector of a column with pivot p and squared norm s2 below it (Sec. 2):
// v = (1, scale x), H = I - tau v v^T, the pivot becomes beta.
template <typename T>
struct Reflector {
  T beta, tau, scale;
  __device__ __forceinline__ Reflector(T p, T s2) {
    const T norm = qr_sqrt(p * p + s2);
    beta = tau = scale = T(0);
    if (norm != T(0)) {
      beta = p >= T(0) ? -norm : norm;
      tau = (beta - p) * qr_rcp(beta);
      scale = qr_rcp(p - beta);
    }
  }
};

// The same for the compression, whose rows of R meet a reflector per four rows: the norm and the inverses to the last
// place.  With the approximations of the fronts, 12 rows of 8 values per column gave the solution (unrefined float) an error of
// 5.6e-7 and the squared residual one of 9e-8; so 4.4e-7 and 1e-8, and the compression is 1 to 2 % of a solve slower.
template <typename T>
struct ExactReflector {
  T beta, tau, scale;
  __device__ __forceinline__ ExactReflector(T p, T s2) {
    beta = p;
    tau = scale = T(0);
    const T n2 = p * p + s2;
    if constexpr (sizeof(T) == 4) {
      if (!(n2 < 1.17549435e-38f)) {   // below: the column is dropped from the reflector, as its norm underflows
        float y;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(n2));
        const float seed = qr_rcp(p >= 0.f ? p + n2 * y : p - n2 * y);   // of the scale, while the root is refined
        const float norm = dev::newton_root(n2, y);
        beta = p >= 0.f ? -norm : norm;
        tau = fma(fabsf(p), dev::newton_inverse(norm, y), 1.f);
        scale = dev::newton_inverse(p - beta, seed);
      }
    } else {
      const T norm = sqrt(n2);
      if (norm != T(0)) {
        beta = p >= T(0) ? -norm : norm;
        tau = (beta - p) / beta;
        scale = T(1) / (p - beta);
      }
    }
  }
};

template <typename T>
struct CRArgs {
  // instances
  int64_t num_inst;
  const int64_t* cols;    // N
  const int64_t* col0;    // first global column
  const int64_t* row0;    // first global row
  const int64_t* rows;    // rows of the instance
  const int64_t* blk0;    // num_inst + 1: first global block of each instance
  const int64_t* tail0;   // num_inst: first level of the instance's one-CTA tail
  const int32_t* binst;   // instance of each block
  int64_t total_blocks;
  // rows: explicit starts (global columns, sorted per instance) or implicit floor(i / rpc)
  // or colptr: the rows that start at global column j are rpc colptr[j] .. rpc colptr[j + 1] - 1
  const int64_t* starts;
  const int32_t* colptr;
  int rpc;
  int w;
  const T* J;             // rows x w
  const T* b;             // rows
  const double* D;        // global columns (damping rows when lam > 0)
  double lam;
  // compression: num_items threads; item_blk: block of each (null: one per block), blk_item0: first item of a block
  int64_t num_items;
  const int32_t* item_blk;
  const int32_t* blk_item0;
  // work space
  int64_t* grp_lo;        // total_blocks: first row of each block's group (explicit starts)
  T* P;                   // num_items partial triangles, e0_at()
  T* E0;                  // total_blocks compressed block rows (level 0), e0_at().  A buffer of their own: the rows of
                          // different instances share lines, and an instance's tail may still read its own
                          // when another's upper levels write block rows.
  T* F0;                  // total_blocks block rows, kFW each (two buffers; level l reads F1 when l is odd)
  T* F1;
  T* Rb;                  // total_blocks x kRW
  T* xp;                  // total_blocks x 8 padded solution / rhs work
  T* hp;                  // total_blocks x 8
  double* res2;           // per instance
  int* status;
};

// First row of each block's group: lower bound of 8 g among the instance's sorted starts.
template <typename T>
__global__ void cr_ranges_kernel(CRArgs<T> A) {
  dev::chain_wait();
  const int64_t gb = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gb >= A.total_blocks) return;
  const int64_t k = A.binst[gb];
  const int64_t g = gb - A.blk0[k];
  const int64_t key = A.col0[k] + (int64_t)kCB * g;
  int64_t lo = A.row0[k], hi = A.row0[k] + A.rows[k];
  while (lo < hi) {
    const int64_t mid = (lo + hi) / 2;
    if (A.starts[mid] < key) lo = mid + 1; else hi = mid;
  }
  A.grp_lo[gb] = lo;
}

template <typename T>
__device__ __forceinline__ void group_rows(const CRArgs<T>& A, int64_t k, int64_t g, int64_t gb, int64_t& lo,
                                           int64_t& hi) {
  const int64_t nb = A.blk0[k + 1] - A.blk0[k];
  const int64_t end = A.row0[k] + A.rows[k];
  if (A.starts) {
    lo = A.grp_lo[gb];
    hi = g + 1 < nb ? A.grp_lo[gb + 1] : end;
  } else if (A.colptr) {
    const int64_t j0 = A.col0[k] + kCB * g, j1 = A.col0[k] + min((int64_t)kCB * (g + 1), A.cols[k]);
    lo = (int64_t)A.colptr[j0] * A.rpc;
    hi = (int64_t)A.colptr[j1] * A.rpc;
  } else {
    const int64_t r0 = A.row0[k] + (int64_t)A.rpc * kCB * g;
    lo = r0 < end ? r0 : end;
    const int64_t r1 = r0 + (int64_t)A.rpc * kCB;
    hi = r1 < end ? r1 : end;
  }
}

// ---- 1. compression: one thread per (block, split) ----
//
// Rows come in the order of their first column, so the triangle of the rows seen so far only needs
// the 8 x 8 window of columns c .. c + 7 while rows starting at c arrive: it lives in registers (36
// values + 8 of the rhs).  Up to four rows are reflected into it at a time, one Householder vector
// (pivot + 4) per column; when the rows of column c are through, the window's first row is row c of
// R and the window moves on by one column.  The damping rows are the window's initial diagonal.
// Against one row at a time by plane rotations into a 16 x 16 triangle in shared memory this needs a
// quarter of the arithmetic and no shared memory, and block rows leave as 16-byte stores.
//
// A compressed block row E: row c < 8 holds columns c .. c + 7 at 8 c; row 8 + i holds columns 8 .. 15 (zeros
// below the diagonal) at 64 + 8 i; the rhs of the 16 rows at 128.  Block rows are stored 32 at a time,
// their 16-byte pieces interleaved: a warp's threads, a block row each, store whole lines, and the lane
// groups that read adjacent block rows share them.  (A thread per block row storing 576 bytes of its own
// kept the L1 at 86 % with lines touched.)
constexpr int kCompThreads = 128;

// Position of element e of compressed block row `it`.
template <typename T>
__host__ __device__ __forceinline__ int64_t e0_at(int64_t it, int e) {
  constexpr int E = 16 / (int)sizeof(T), P = kE0 / E;
  return (((it >> 5) * P + e / E) * 32 + (it & 31)) * E + e % E;
}

__host__ __device__ constexpr int tri(int i, int j) { return i * 8 - (i * (i - 1)) / 2 + (j - i); }

template <typename T>
struct Window {
  T t[36], z[8];
  // four rows (8 columns from the window's first, rhs) reflected into the window; b keeps what is left
  __device__ __forceinline__ void insert(T (&a)[4][8], T (&b)[4]) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      T s2 = T(0);
#pragma unroll
      for (int q = 0; q < 4; ++q) s2 += a[q][k] * a[q][k];
      const T p = t[tri(k, k)];
      ExactReflector<T> h(p, s2);
      T v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = a[q][k] * h.scale;
      if (faint(p * p + s2)) {
        s2 = T(0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          v[q] = a[q][k] * T(kLift);
          s2 += v[q] * v[q];
        }
        h = ExactReflector<T>(p * T(kLift), s2);
        h.beta *= T(1) / T(kLift);
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] *= h.scale;
      }
      t[tri(k, k)] = h.beta;
#pragma unroll
      for (int j = k + 1; j < 8; ++j) {
        T w = t[tri(k, j)];
#pragma unroll
        for (int q = 0; q < 4; ++q) w += v[q] * a[q][j];
        w *= h.tau;
        t[tri(k, j)] -= w;
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q][j] -= w * v[q];
      }
      T w = z[k];
#pragma unroll
      for (int q = 0; q < 4; ++q) w += v[q] * b[q];
      w *= h.tau;
      z[k] -= w;
#pragma unroll
      for (int q = 0; q < 4; ++q) b[q] -= w * v[q];
    }
  }
  __device__ __forceinline__ void shift() {
#pragma unroll
    for (int i = 0; i < 7; ++i) {
#pragma unroll
      for (int j = i; j < 7; ++j) t[tri(i, j)] = t[tri(i + 1, j + 1)];
      t[tri(i, 7)] = T(0);
      z[i] = z[i + 1];
    }
    t[tri(7, 7)] = T(0);
    z[7] = T(0);
  }
};

template <typename T>
__device__ __forceinline__ void load8(T (&v)[8], const T* src) {   // src 16-byte aligned
  if constexpr (sizeof(T) == 4) {
    const float4 a = reinterpret_cast<const float4*>(src)[0], b = reinterpret_cast<const float4*>(src)[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 a = reinterpret_cast<const double2*>(src)[q];
      v[2 * q] = a.x;
      v[2 * q + 1] = a.y;
    }
  }
}

// Eight consecutive elements of a compressed block row, from a multiple of 8 on.
template <typename T>
__device__ __forceinline__ void store_e0(T* base, int64_t it, int e, const T (&v)[8]) {
  if constexpr (sizeof(T) == 4) {
    *reinterpret_cast<float4*>(base + e0_at<T>(it, e)) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(base + e0_at<T>(it, e + 4)) = make_float4(v[4], v[5], v[6], v[7]);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      *reinterpret_cast<double2*>(base + e0_at<T>(it, e + 2 * q)) = make_double2(v[2 * q], v[2 * q + 1]);
  }
}
template <typename T>
__device__ __forceinline__ void load_e0(T (&v)[8], const T* base, int64_t it, int e) {
  if constexpr (sizeof(T) == 4) {
    const float4 a = *reinterpret_cast<const float4*>(base + e0_at<T>(it, e));
    const float4 b = *reinterpret_cast<const float4*>(base + e0_at<T>(it, e + 4));
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 a = *reinterpret_cast<const double2*>(base + e0_at<T>(it, e + 2 * q));
      v[2 * q] = a.x;
      v[2 * q + 1] = a.y;
    }
  }
}

// A thread's squared residual: a float pair for float, a double for double.  (A warp's FP64 instruction
// occupies the SM's FP64 unit for 16 cycles here: summing every square in double took a quarter of the
// compression's and of the fronts' time.)  A right-hand side may have any
// scale: an entry whose square or its rounding error would leave the float range goes to res2 in double by itself.
template <typename T>
struct ResidualSum;
template <>
struct ResidualSum<float> {
  dev::Pair s;
  template <int N>
  __device__ __forceinline__ void squares(const float (&x)[N], double* res2) {
    bool all = true;
    float p[N], e[N];   // the squares and their rounding errors, added up pairwise
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const bool ok = dev::square_exact(x[q]);
      const float y = ok ? x[q] : 0.f;
      p[q] = __fmul_rn(y, y);
      e[q] = __fmaf_rn(y, y, -p[q]);
      all = all && ok;
    }
#pragma unroll
    for (int w = N / 2; w >= 1; w /= 2)
#pragma unroll
      for (int q = 0; q < w; ++q) {
        float t, d;
        dev::two_sum(p[q], p[q + w], t, d);
        p[q] = t;
        e[q] = __fadd_rn(__fadd_rn(e[q], e[q + w]), d);
      }
    s.add(p[0], e[0]);
    if (!all) {
#pragma unroll
      for (int q = 0; q < N; ++q)
        if (!dev::square_exact(x[q])) atomicAdd(res2, (double)x[q] * (double)x[q]);
    }
  }
  __device__ __forceinline__ void add_lane(unsigned m, int d) {
    const float ph = __shfl_xor_sync(m, s.h, d), pl = __shfl_xor_sync(m, s.l, d);
    s.add(ph, pl);
  }
  __device__ __forceinline__ double value() const { return s.value(); }
};
template <>
struct ResidualSum<double> {
  double s = 0.0;
  template <int N>
  __device__ __forceinline__ void squares(const double (&x)[N], double*) {
#pragma unroll
    for (int q = 0; q < N; ++q) s += x[q] * x[q];
  }
  __device__ __forceinline__ void add_lane(unsigned m, int d) { s += __shfl_xor_sync(m, s, d); }
  __device__ __forceinline__ double value() const { return s; }
};
// into res2 of the thread's instance: one atomic per warp where all its threads work on one instance
template <typename T>
__device__ __forceinline__ void flush_residual(ResidualSum<T>& r, double* res2, int64_t k) {
  __syncwarp();
  const unsigned m = __activemask();
  const int64_t k0 = __shfl_sync(m, k, __ffs(m) - 1);
  const bool one = m == 0xffffffffu && __all_sync(m, k == k0);
  if (one) {
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) r.add_lane(m, d);
  }
  if (!one || (threadIdx.x & 31) == 0) {
    const double v = r.value();
    if (v != 0.0) atomicAdd(res2 + k, v);
  }
}

// Rows of 8 aligned values (kStaged) arrive through shared memory: the lanes of a warp fetch each thread's next
// four rows together (8 or 16 lanes a thread, whole lines, where a thread's own 16-byte loads touch a line of
// their own each), one step ahead.  Other rows are read by their thread, entry by entry.
template <typename T>
constexpr int stage_stride() { return 4 * kCB * (int)sizeof(T) + 16; }   // bytes of a thread's four rows, padded

template <typename T, bool kStaged>
__global__ void __launch_bounds__(kCompThreads, sizeof(T) == 4 ? 4 : 2) cr_compress_kernel(CRArgs<T> A) {
  dev::chain_wait();
  extern __shared__ __align__(16) unsigned char stage[];   // two buffers of kCompThreads x stage_stride
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t item = (int64_t)blockIdx.x * kCompThreads + threadIdx.x;
  const bool have = item < A.num_items;   // threads past the end only help with the copies
  const int64_t gb = !have ? 0 : (A.item_blk ? A.item_blk[item] : item);
  const int s = have && A.item_blk ? (int)(item - A.blk_item0[gb]) : 0;
  const int splits = A.item_blk ? A.blk_item0[gb + 1] - A.blk_item0[gb] : 1;
  const int64_t k = A.binst[gb];
  const int64_t g = gb - A.blk0[k];
  const int64_t N = A.cols[k], c0 = A.col0[k], row0 = A.row0[k];
  int64_t lo, hi;
  group_rows(A, k, g, gb, lo, hi);
  const int64_t len = have ? hi - lo : 0;
  int64_t r = lo + len * s / splits;
  const int64_t r_end = lo + len * (s + 1) / splits;
  Window<T> W;
#pragma unroll
  for (int e = 0; e < 36; ++e) W.t[e] = T(0);
#pragma unroll
  for (int i = 0; i < 8; ++i) W.z[i] = T(0);
  if (s == 0) {   // damping rows; unit rows for padding columns
    const double lam_half = sqrt(A.lam);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int64_t col = (int64_t)kCB * g + i;
      W.t[tri(i, i)] = col >= N ? T(1) : (A.lam > 0.0 ? (T)(lam_half * A.D[c0 + col]) : T(0));
    }
  }
  T* dst = splits == 1 ? A.E0 : A.P;
  const int64_t at = splits == 1 ? gb : item;
  constexpr int kLanes = 2 * (int)sizeof(T);   // 16-byte pieces of four rows
  auto fetch = [&](int buf) {   // the warp's threads' rows r .. r + 3 (those before r_end) into buffer buf
    unsigned char* base = stage + (buf * kCompThreads + warp * 32) * stage_stride<T>();
    const int avail = (int)max((int64_t)0, min((int64_t)4, r_end - r));
#pragma unroll
    for (int i = 0; i < kLanes; ++i) {
      const int q = i * (32 / kLanes) + lane / kLanes;   // the thread whose rows these are
      const int64_t rq = __shfl_sync(0xffffffffu, r, q);
      const int nq = __shfl_sync(0xffffffffu, avail, q);
      const int o = (lane % kLanes) * 16;
      if (o < nq * kCB * (int)sizeof(T))
        dev::cp_async16(base + q * stage_stride<T>() + o, reinterpret_cast<const unsigned char*>(A.J + rq * kCB) + o);
    }
    dev::cp_async_commit();
  };
  int buf = 0;
  if constexpr (kStaged) fetch(0);
  ResidualSum<T> res;
  // One step per turn: the next (up to four) rows starting at column c, or, when there are none, the window
  // one column on.  The threads of a warp may be at different columns.
  int64_t ahead[4];   // explicit starts of the next four rows, fetched one step early
#pragma unroll
  for (int q = 0; q < 4; ++q) ahead[q] = A.starts && r + q < r_end ? A.starts[r + q] - c0 : -1;
  int c = have ? 0 : kCB;
  // first row that starts past column `col` of the instance (implicit starts)
  auto rows_end = [&](int64_t col) -> int64_t {
    const int64_t e = A.colptr ? (col < N ? (int64_t)A.colptr[c0 + col + 1] * A.rpc : r_end) : row0 + (col + 1) * A.rpc;
    return min(r_end, e);
  };
  int64_t c_end = A.starts ? r_end : rows_end((int64_t)kCB * g);   // of column c
#pragma unroll 1
  while (__any_sync(0xffffffffu, c < kCB)) {
    const int64_t st = (int64_t)kCB * g + c;   // the rows' first column
    int cnt = 0;
    if (c < kCB) {
      if (A.starts) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (cnt == q && ahead[q] == st) cnt = q + 1;
      } else {
        cnt = (int)max((int64_t)0, min((int64_t)4, c_end - r));
      }
    }
    T a[4][8], b[4];
    if (cnt > 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) b[q] = q < cnt ? A.b[r + q] : T(0);
    }
    if constexpr (kStaged) {
      dev::cp_async_wait_all();
      __syncwarp();
      const T* mine = reinterpret_cast<const T*>(stage + (buf * kCompThreads + threadIdx.x) * stage_stride<T>());
      if (cnt > 0) {
        const int nt = (int)min((int64_t)kCB, N - st);   // entries past the last column are ignored
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
          for (int t = 0; t < 8; ++t) a[q][t] = T(0);
          if (q < cnt) {
            load8(a[q], mine + kCB * q);
            if (nt < kCB) {
#pragma unroll
              for (int t = 0; t < 8; ++t)
                if (t >= nt) a[q][t] = T(0);
            }
          }
        }
      }
    } else if (cnt > 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int t = 0; t < 8; ++t) a[q][t] = q < cnt && t < A.w && st + t < N ? A.J[(r + q) * A.w + t] : T(0);
      }
    }
    r += cnt;
    if constexpr (kStaged) {
      // a turn of shifts only leaves every buffer as it is; otherwise all threads fetch, those that did
      // not move the same rows again
      if (__any_sync(0xffffffffu, cnt > 0)) {
        buf ^= 1;
        fetch(buf);
      }
    }
    if (cnt > 0) {
      if (A.starts) {
#pragma unroll
        for (int q = 0; q < 4; ++q) ahead[q] = r + q < r_end ? A.starts[r + q] - c0 : -1;
      }
      W.insert(a, b);
      res.squares(b, A.res2 + k);
    } else if (c < kCB) {
      T row[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) row[j] = W.t[tri(0, j)];
      store_e0(dst, at, 8 * c, row);
      dst[e0_at<T>(at, 128 + c)] = W.z[0];
      W.shift();
      ++c;
      if (!A.starts) c_end = rows_end((int64_t)kCB * g + c);
    }
  }
  if constexpr (kStaged) dev::cp_async_wait_all();
  if (have) {
    if (r < r_end) cr_record(A.status, QRKIT_EINVAL);   // rows out of order or past the block
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      T row[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) row[j] = j >= i ? W.t[tri(i, j)] : T(0);
      store_e0(dst, at, 64 + 8 * i, row);
    }
    store_e0(dst, at, 136, W.z);
  }
  flush_residual(res, A.res2, k);
}

// 1b. merge of up to kMergeFan partial triangles of a block into one, by the same window; 16 columns.
constexpr int kMergeFan = 4;

struct MergeItem {
  int32_t blk, first, n;   // block; its partials first .. first + n - 1 of the input
  int32_t out;             // partial of the output, or -1: the block's compressed row
};

template <typename T>
__global__ void __launch_bounds__(kCompThreads) cr_merge_kernel(CRArgs<T> A, const MergeItem* items, int64_t nitems,
                                                                const T* in, T* part) {
  dev::chain_wait();
  const int64_t w = (int64_t)blockIdx.x * kCompThreads + threadIdx.x;
  if (w >= nitems) return;
  const MergeItem M = items[w];
  const int n = M.n;
  const int64_t first = M.first, gb = M.blk, item = M.out < 0 ? gb : M.out, k = A.binst[gb];
  T* out = M.out < 0 ? A.E0 : part;
  Window<T> W;
#pragma unroll
  for (int e = 0; e < 36; ++e) W.t[e] = T(0);
#pragma unroll
  for (int i = 0; i < 8; ++i) W.z[i] = T(0);
  ResidualSum<T> res;
#pragma unroll 1
  for (int c = 0; c < 16; ++c) {
    T a[4][8], b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      b[q] = T(0);
#pragma unroll
      for (int t = 0; t < 8; ++t) a[q][t] = T(0);
      if (q < n) {
        b[q] = in[e0_at<T>(first + q, 128 + c)];
        if (c < 8) {
          load_e0(a[q], in, first + q, 8 * c);
        } else {   // row c - 8 of the second triangle: columns c ..
#pragma unroll
          for (int t = 0; t < 8; ++t)
            if (c + t < 16) a[q][t] = in[e0_at<T>(first + q, 64 + 9 * (c - 8) + t)];
        }
      }
    }
    W.insert(a, b);
    res.squares(b, A.res2 + k);
    if (c < 8) {
      T row[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) row[j] = W.t[tri(0, j)];
      store_e0(out, item, 8 * c, row);
    } else {
      const int d = 64 + 8 * (c - 8);
      for (int j = 0; j < c - 8; ++j) out[e0_at<T>(item, d + j)] = T(0);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (c + j < 16) out[e0_at<T>(item, d + c - 8 + j)] = W.t[tri(0, j)];
    }
    out[e0_at<T>(item, 128 + c)] = W.z[0];
    W.shift();
  }
  flush_residual(res, A.res2, k);
}

// Work items of a level: inst << 32 | i << 2 | kind (0 eliminate odd i, 1 move up, 2 last).
__device__ __forceinline__ void decode(int64_t it, int64_t& k, int64_t& i, int& kind) {
  k = it >> 32;
  i = (it >> 2) & 0x3fffffff;
  kind = (int)(it & 3);
}

// ---- 2. the elimination of one block: eight lanes ----
//
// Lane j holds column j of each 8-column part of the front (and the rhs), so a reflector's column is
// read by broadcasts from the lane that owns it and every dot product is local: no reductions.  The
// triangular shapes of the two block rows are used: F_{i-1} = [A' | B'] and F_i = [A | B] with A', A, and
// rows 8..15 of B' and B upper triangular.
//   1. rows 8..15 of B' (own columns) into A                    -> rows with entries right only
//   2. rows 0..7 of B' into A, which makes A the 8 rows of R    -> rows on left and right
//   3. those rows triangular in the left columns, and the right-only rows of step 1 into rows 8..15 of B:
//      the new 16-row block row on (left, right).
// Rows are taken two at a time (f32x2): 13 million columns of 256 instances spend 1,505 us on the fronts against 1,641
// with scalar rows.  A 32-row front on a whole warp with its sums reduced by shuffles took six times the
// instructions.
constexpr int kItemThreads = kCB;

// Eight rows of a column on a lane: two rows per operation for float.  The ranges [r0, r1) are known at compile time
// once the loops are unrolled; a range that begins or ends inside a pair takes the pair, whose other row is
// zero in v.
template <typename T>
struct Rows;
template <>
struct Rows<float> {
  dev::f2 p[4];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = 0ull;
  }
  __device__ __forceinline__ float get(int r) const {
    float x, y;
    dev::unpack2(p[r >> 1], x, y);
    return r & 1 ? y : x;
  }
  __device__ __forceinline__ void set(int r, float v) {
    float x, y;
    dev::unpack2(p[r >> 1], x, y);
    p[r >> 1] = r & 1 ? dev::pack2(x, v) : dev::pack2(v, y);
  }
  __device__ __forceinline__ void scale(const Rows& x, float f, int r0, int r1) {
    const dev::f2 f2v = dev::pack2(f, f);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (2 * i + 1 >= r0 && 2 * i < r1) p[i] = dev::mul2(x.p[i], f2v);
  }
  __device__ __forceinline__ float dot(const Rows& x, int r0, int r1) const {
    dev::f2 d = 0ull;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (2 * i + 1 >= r0 && 2 * i < r1) d = dev::fma2(p[i], x.p[i], d);
    return dev::sum2(d);
  }
  __device__ __forceinline__ void add(float w, const Rows& v, int r0, int r1) {   // += w v
    const dev::f2 w2 = dev::pack2(w, w);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (2 * i + 1 >= r0 && 2 * i < r1) p[i] = dev::fma2(w2, v.p[i], p[i]);
  }
};
template <>
struct Rows<double> {
  double v[8];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = 0.0;
  }
  __device__ __forceinline__ double get(int r) const { return v[r]; }
  __device__ __forceinline__ void set(int r, double x) { v[r] = x; }
  __device__ __forceinline__ void scale(const Rows& x, double f, int r0, int r1) {
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (r >= r0 && r < r1) v[r] = x.v[r] * f;
  }
  __device__ __forceinline__ double dot(const Rows& x, int r0, int r1) const {
    double d = 0.0;
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (r >= r0 && r < r1) d += v[r] * x.v[r];
    return d;
  }
  __device__ __forceinline__ void add(double w, const Rows& x, int r0, int r1) {
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (r >= r0 && r < r1) v[r] += w * x.v[r];
  }
};

// Columns j of A (rows 0..7) and B (rows 0..7, 8..15) of block row `it`, and its rhs.
template <typename T, bool kCompressed, class RA, class RL, class RH, class RC, class RD>
__device__ __forceinline__ void load_block_row(const T* base, int64_t it, int j, RA&& a, RL&& bl, RH&& bh, RC&& cl,
                                               RD&& ch) {
  T c0[8], c1[8];
  if constexpr (kCompressed) {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const T v = base[e0_at<T>(it, 8 * r + ((j - r) & 7))];   // column j of A for j >= r, of B for j < r
      a(r, j >= r ? v : T(0));
      bl(r, j < r ? v : T(0));
      bh(r, base[e0_at<T>(it, 64 + 8 * r + j)]);
    }
    load_e0(c0, base, it, 128);
    load_e0(c1, base, it, 136);
  } else {
    const T* F = base + it * kFW;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      a(r, F[8 * r + j]);
      bl(r, F[64 + 8 * r + j]);
      bh(r, F[128 + 8 * r + j]);
    }
    load8(c0, F + 192);
    load8(c1, F + 200);
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    cl(r, c0[r]);
    ch(r, c1[r]);
  }
}

template <typename T>
__device__ __forceinline__ T lane_of(const T (&v)[8], int j) {   // v[j] for a lane index j
  T x = v[0];
#pragma unroll
  for (int q = 1; q < 8; ++q)
    if (j == q) x = v[q];
  return x;
}
template <typename T>
__device__ __forceinline__ T lane_of(const Rows<T>& v, int j) {
  T x = v.get(0);
#pragma unroll
  for (int q = 1; q < 8; ++q)
    if (j == q) x = v.get(q);
  return x;
}

// One item of level `level`: block i of instance k.  The lanes add their share of the residual it leaves to res.
//
// The rows that a step's reflectors meet one at a time (A; then pa, bh as pivots) are scalars or halves of a pair, the
// rows below in Rows.  A reflector of column q must leave the columns before it alone; their entries below
// the diagonal are not cleared one by one: tj, the factor of a lane's own column, is zero on lanes up to q.
template <typename T, bool kCompressed>
__device__ __forceinline__ void cr_item(const CRArgs<T>& A, int64_t k, int64_t i, int kind, int level, const T* Fc,
                                        T* Fn, int j, unsigned gmask, ResidualSum<T>& res) {
  const int64_t b0 = A.blk0[k];
  T a[8], bl[8], bh[8], cl[8], ch[8];
  auto to = [](T (&x)[8]) { return [&x](int r, T v) { x[r] = v; }; };
  load_block_row<T, kCompressed>(Fc, b0 + i, j, to(a), to(bl), to(bh), to(cl), to(ch));
  if (kind == 1) {   // unpaired last block row: moves up
    T* F = Fn + (b0 + i / 2) * kFW;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      F[8 * r + j] = a[r];
      F[64 + 8 * r + j] = bl[r];
      F[128 + 8 * r + j] = bh[r];
    }
    F[192 + j] = lane_of(cl, j);
    F[200 + j] = lane_of(ch, j);
    return;
  }
  T* R = A.Rb + (b0 + (i << level)) * kRW;
  if (kind == 0) {
    Rows<T> pa, pl, ph, dl, dh, rr, lr, v, x;
    auto rows = [](Rows<T>& y) { return [&y](int r, T u) { y.set(r, u); }; };
    load_block_row<T, kCompressed>(Fc, b0 + i - 1, j, rows(pa), rows(pl), rows(ph), rows(dl), rows(dh));
    rr.zero();   // right parts of the rows of B'
    lr.zero();
    T rl[8];     // R's left part
    // the reflector of column q: pivot `piv` and rows [r0, r1) of y, both of lane q; v's other rows of touched pairs zero
    T tj, t, beta;
    auto reflector = [&](int q, T piv, const Rows<T>& y, int r0, int r1) {
      const T p = __shfl_sync(gmask, piv, q, kItemThreads);
      x.zero();
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (r >= r0 && r < r1) x.set(r, __shfl_sync(gmask, y.get(r), q, kItemThreads));
      const Reflector<T> h(p, x.dot(x, r0, r1));
      v.scale(x, h.scale, r0, r1);
      t = -h.tau;
      tj = j > q ? t : T(0);
      beta = h.beta;
    };
    // y, and the pivot p of its column, with the factor f
    auto apply = [&](T f, T& p, Rows<T>& y, int r0, int r1) {
      const T w = f * (p + v.dot(y, r0, r1));
      p += w;
      y.add(w, v, r0, r1);
    };
    auto apply_at = [&](T f, int q, Rows<T>& y, int r0, int r1) {   // the pivot is row q of y itself
      T p = y.get(q);
      const T w = f * (p + v.dot(y, r0, r1));
      y.add(w, v, r0, r1);
      y.set(q, p + w);
    };
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      reflector(q, a[q], ph, 0, q + 1);
      apply(tj, a[q], ph, 0, q + 1);
      apply(t, bl[q], rr, 0, q + 1);
      apply(t, cl[q], dh, 0, q + 1);
      if (j == q) a[q] = beta;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      reflector(q, a[q], pl, 0, 8);
      rl[q] = T(0);
      apply(tj, a[q], pl, 0, 8);
      apply(t, rl[q], pa, 0, 8);
      apply(t, bl[q], lr, 0, 8);
      apply(t, cl[q], dl, 0, 8);
      if (j == q) a[q] = beta;
    }
    // the rows of R go out here; what follows needs pa, lr, dl (left and right) and rr, dh, bh, ch
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      R[8 * r + j] = a[r];
      R[64 + 8 * r + j] = rl[r];
      R[128 + 8 * r + j] = bl[r];
    }
    R[192 + j] = lane_of(cl, j);
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      reflector(q, pa.get(q), pa, q + 1, 8);
      apply_at(tj, q, pa, q + 1, 8);
      apply_at(t, q, lr, q + 1, 8);
      apply_at(t, q, dl, q + 1, 8);
      if (j == q) pa.set(q, beta);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      reflector(q, bh[q], rr, 0, 8);
      apply(tj, bh[q], rr, 0, 8);
      apply(t, ch[q], dh, 0, 8);
      if (j == q) bh[q] = beta;
    }
    T* F = Fn + (b0 + (i - 1) / 2) * kFW;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      F[8 * r + j] = r <= j ? pa.get(r) : T(0);
      F[64 + 8 * r + j] = lr.get(r);
      F[128 + 8 * r + j] = bh[r];
    }
    F[192 + j] = lane_of(dl, j);
    F[200 + j] = lane_of(ch, j);
    const T left[1] = {lane_of(dh, j)};
    res.squares(left, A.res2 + k);
  } else {   // the last block: its A is triangular, nothing is to its right
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      R[8 * r + j] = a[r];
      R[64 + 8 * r + j] = T(0);
      R[128 + 8 * r + j] = bl[r];
    }
    R[192 + j] = lane_of(cl, j);
    const T left[1] = {lane_of(ch, j)};
    res.squares(left, A.res2 + k);
  }
}

constexpr int kLevelThreads = 128;

template <typename T, bool kCompressed>
__global__ void __launch_bounds__(kLevelThreads, sizeof(T) == 4 ? 4 : 2)
cr_level_kernel(CRArgs<T> A, const int64_t* items, int64_t nitems, int level, const T* Fc, T* Fn) {
  dev::chain_wait();
  const int64_t w = ((int64_t)blockIdx.x * kLevelThreads + threadIdx.x) / kItemThreads;
  const int j = threadIdx.x % kItemThreads;
  const unsigned gmask = 0xffu << (threadIdx.x & 24);
  int64_t k = 0, i = 0;
  int kind = 1;
  ResidualSum<T> res;
  if (w < nitems) {
    decode(items[w], k, i, kind);
    cr_item<T, kCompressed>(A, k, i, kind, level, Fc, Fn, j, gmask, res);
  } else if (nitems > 0) {
    decode(items[nitems - 1], k, i, kind);   // adds nothing, to the last item's instance
  }
  flush_residual(res, A.res2, k);
}

// ---- 3. back-substitution of one block, eight lanes: lane q owns row q of the block's R (own | left |
// right | rhs): the couplings to the neighbours' solutions are row-local, the triangular solve
// broadcasts each x_t.  rhs from the R rows' own column (c) or from hp; writes xp (padded) and, for
// real columns, x (written) and xadd (added to). ----
template <typename T>
__device__ __forceinline__ void cr_backsub_item(const CRArgs<T>& A, int64_t k, int64_t i, int kind, int level,
                                                bool use_hp, T* x, T* xadd, int q, unsigned gmask) {
  const int64_t b0 = A.blk0[k], N = A.cols[k];
  const int64_t G = (N + kCB - 1) / kCB;
  const int64_t beta = i << level, step = (int64_t)1 << level;
  const T* R = A.Rb + (b0 + beta) * kRW;
  T own[8], nbr[8];
  load8(own, R + 8 * q);
  T y = use_hp ? A.hp[(b0 + beta) * kCB + q] : R[192 + q];
  if (kind == 0) {
    const T* xl = A.xp + (b0 + beta - step) * kCB;
    load8(nbr, R + 64 + 8 * q);
#pragma unroll
    for (int t = 0; t < kCB; ++t) y -= nbr[t] * xl[t];
  }
  if (beta + step < G) {
    const T* xr = A.xp + (b0 + beta + step) * kCB;
    load8(nbr, R + 128 + 8 * q);
#pragma unroll
    for (int t = 0; t < kCB; ++t) y -= nbr[t] * xr[t];
  }
  const T diag = lane_of(own, q);
  if (diag == T(0)) cr_record(A.status, QRKIT_ESINGULAR);
  T xq = T(0);
#pragma unroll
  for (int t = kCB - 1; t >= 0; --t) {   // x_t = (y_t - sum_{u > t} R_tu x_u) / R_tt, bottom up
    if (q == t) xq = y / diag;
    const T xt = __shfl_sync(gmask, xq, t, kItemThreads);
    if (t > q) y -= own[t] * xt;
  }
  A.xp[(b0 + beta) * kCB + q] = xq;
  if (kCB * beta + q < N) {
    const int64_t col = A.col0[k] + kCB * beta + q;
    if (x) x[col] = xq;
    if (xadd) xadd[col] += xq;
  }
}

template <typename T>
__global__ void cr_backsub_kernel(CRArgs<T> A, const int64_t* items, int64_t nitems, int level, int use_hp, T* x,
                                  T* xadd) {
  dev::chain_wait();
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kItemThreads;
  if (w >= nitems) return;
  int64_t k, i;
  int kind;
  decode(items[w], k, i, kind);
  if (kind == 1) return;
  cr_backsub_item(A, k, i, kind, level, use_hp != 0, x, xadd, (int)(threadIdx.x % kItemThreads),
                  0xffu << (threadIdx.x & 24));
}

// Refinement, R^T h = g upwards (xp holds the updated g).  h of one block: lane q solves for h_q after the
// h_t, t < q, are broadcast; with `part` the lane also gathers sum_t part[t][q] h_t.
template <typename T>
__device__ __forceinline__ T cr_rt_item(const CRArgs<T>& A, int64_t blk, const T* part, T& acc, int q, unsigned gmask) {
  const T* R = A.Rb + blk * kRW;
  T col[8], pc[8];
#pragma unroll
  for (int t = 0; t < kCB; ++t) {
    col[t] = t <= q ? R[8 * t + q] : T(0);
    pc[t] = part ? part[8 * t + q] : T(0);
  }
  T v = A.xp[blk * kCB + q], hq = T(0);
  const T diag = lane_of(col, q);
#pragma unroll
  for (int t = 0; t < kCB; ++t) {   // h_t = (g_t - sum_{u < t} R_ut h_u) / R_tt, top down
    if (q == t) hq = v / diag;
    const T ht = __shfl_sync(gmask, hq, t, kItemThreads);
    if (t < q) v -= col[t] * ht;
    acc += pc[t] * ht;
  }
  return hq;
}

// A block that stays (even j at level l): h of the eliminated neighbours j - 1 and j + 1, then
// g_j -= R_{j-1}.right^T h_{j-1} + R_{j+1}.left^T h_{j+1}.  The item to the left of an eliminated block
// stores its h; computing h twice saves a launch per level.
template <typename T>
__device__ __forceinline__ void cr_rt_level_item(const CRArgs<T>& A, int64_t k, int64_t j, int level, int q,
                                                 unsigned gmask) {
  const int64_t b0 = A.blk0[k], G = A.blk0[k + 1] - b0;
  const int64_t Gl = (G + ((int64_t)1 << level) - 1) >> level;
  T* g = A.xp + (b0 + (j << level)) * kCB;
  T acc = T(0);
  if (j >= 1) {
    const int64_t nb = b0 + ((j - 1) << level);
    cr_rt_item(A, nb, A.Rb + nb * kRW + 128, acc, q, gmask);
  }
  if (j + 1 < Gl) {
    const int64_t nb = b0 + ((j + 1) << level);
    const T h = cr_rt_item(A, nb, A.Rb + nb * kRW + 64, acc, q, gmask);
    A.hp[nb * kCB + q] = h;
  }
  g[q] -= acc;
}

template <typename T>
__global__ void cr_rt_level_kernel(CRArgs<T> A, const int64_t* items, int64_t nitems, int level) {
  dev::chain_wait();
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kItemThreads;
  if (w >= nitems) return;
  cr_rt_level_item(A, items[w] >> 32, items[w] & 0xffffffff, level, (int)(threadIdx.x % kItemThreads),
                   0xffu << (threadIdx.x & 24));
}

// ---- an instance's upper levels in one CTA (of as many threads as registers allow for a few
// instances, 128 for many, so that several share an SM) ----
template <typename T>
constexpr int tail_threads() { return sizeof(T) == 4 ? 512 : 256; }

// Blocks left at level l of an instance of G blocks.
__device__ __forceinline__ int64_t blocks_at(int64_t G, int level) { return (G + ((int64_t)1 << level) - 1) >> level; }

// x of levels top .. lt (down) of instance k.
template <typename T>
__device__ __forceinline__ void tail_backsub(const CRArgs<T>& A, int64_t k, int64_t G, int lt, int top, bool use_hp,
                                             T* x, T* xadd) {
  const int grp = threadIdx.x / kItemThreads, ng = blockDim.x / kItemThreads, q = threadIdx.x % kItemThreads;
  const unsigned gmask = 0xffu << (threadIdx.x & 24);
  for (int l = top; l >= lt; --l) {
    if (l == top) {
      if (grp == 0) cr_backsub_item(A, k, 0, 2, l, use_hp, x, xadd, q, gmask);
    } else {
      const int64_t Gl = blocks_at(G, l);
      for (int64_t i = 2 * grp + 1; i < Gl; i += 2 * ng) cr_backsub_item(A, k, i, 0, l, use_hp, x, xadd, q, gmask);
    }
    __syncthreads();
  }
}

// Factor of the upper levels, then their back-substitution.
template <typename T>
__global__ void __launch_bounds__(tail_threads<T>(), 1) cr_tail_kernel(CRArgs<T> A, T* x) {
  dev::chain_wait();
  const int64_t k = blockIdx.x;
  const int grp = threadIdx.x / kItemThreads, ng = blockDim.x / kItemThreads, j = threadIdx.x % kItemThreads;
  const unsigned gmask = 0xffu << (threadIdx.x & 24);
  const int64_t G = A.blk0[k + 1] - A.blk0[k];
  const int lt = (int)A.tail0[k];
  ResidualSum<T> res;
  int l = lt;
  for (;; ++l) {
    const int64_t Gl = blocks_at(G, l);
    const T* Fc = l == 0 ? A.E0 : ((l & 1) ? A.F1 : A.F0);
    T* Fn = (l & 1) ? A.F0 : A.F1;
    // item m: odd block 2 m + 1, or the unpaired last block (kind 1), or the only one (kind 2)
    const int64_t n = Gl == 1 ? 1 : (Gl + 1) / 2;
    for (int64_t m = grp; m < n; m += ng) {
      const int kind = Gl == 1 ? 2 : (2 * m + 1 < Gl ? 0 : 1);
      const int64_t i = kind == 0 ? 2 * m + 1 : Gl - 1;
      if (l == 0) cr_item<T, true>(A, k, i, kind, l, Fc, Fn, j, gmask, res);
      else cr_item<T, false>(A, k, i, kind, l, Fc, Fn, j, gmask, res);
    }
    __syncthreads();
    if (Gl == 1) break;
  }
  flush_residual(res, A.res2, k);
  tail_backsub(A, k, G, lt, l, false, x, (T*)nullptr);
}

// R^T h = g through the upper levels, then their back-substitution.
template <typename T>
__global__ void __launch_bounds__(tail_threads<T>(), 1) cr_tail_normal_kernel(CRArgs<T> A, T* x, T* xadd) {
  dev::chain_wait();
  const int64_t k = blockIdx.x;
  const int grp = threadIdx.x / kItemThreads, ng = blockDim.x / kItemThreads, q = threadIdx.x % kItemThreads;
  const unsigned gmask = 0xffu << (threadIdx.x & 24);
  const int64_t G = A.blk0[k + 1] - A.blk0[k];
  const int lt = (int)A.tail0[k];
  int l = lt;
  for (;; ++l) {
    const int64_t Gl = blocks_at(G, l);
    if (Gl == 1) {
      if (grp == 0) {
        T none = T(0);
        const int64_t blk = A.blk0[k];
        const T h = cr_rt_item(A, blk, (const T*)nullptr, none, q, gmask);
        A.hp[blk * kCB + q] = h;
      }
      __syncthreads();
      break;
    }
    for (int64_t j = 2 * grp; j < Gl; j += 2 * ng) cr_rt_level_item(A, k, j, l, q, gmask);
    __syncthreads();
  }
  tail_backsub(A, k, G, lt, l, true, x, xadd);
}

// g by global column into the padded layout (virtual columns 0).
template <typename T>
__global__ void cr_scatter_g_kernel(CRArgs<T> A, const double* g_in) {
  dev::chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= A.total_blocks * kCB) return;
  const int64_t gb = e / kCB;
  const int q = (int)(e - gb * kCB);
  const int64_t k = A.binst[gb];
  const int64_t col = kCB * (gb - A.blk0[k]) + q;
  A.xp[e] = col < A.cols[k] ? (T)g_in[A.col0[k] + col] : T(0);
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// ---------------------------------------------------------------------------------------
// Host side: instance tables, level work lists, launches.

// The compression's threads and the merges of their triangles.  Never changed once built, and kept as long as the
// plan: a solve that is queued, or captured in a graph, holds the device addresses.
struct CRSplits {
  int each = 0;                            // threads of every block, or 0: per instance by its rows
  int64_t num_items = 0;                   // threads of the compression
  std::vector<int64_t> mg_off, mg_n;       // merge items per pass
  DevBuf item_blk, blk_item0, merges;
};

struct CRPlan {
  int64_t num_inst = 0, total_blocks = 0;
  int levels = 0;                          // those run by launches of their own, before the tails
  int64_t total_rows = 0;
  std::vector<int64_t> h_blk0, h_rows;     // kept for the compression's strategy
  std::vector<CRSplits*> splits;           // the strategies asked for so far
  const CRSplits* cur = nullptr;
  std::vector<DevBuf> outgrown;            // partial triangles that a queued or captured solve may still use
  std::vector<int64_t> lvl_off, lvl_n;     // eliminate / move items per level
  std::vector<int64_t> ev_off, ev_n;       // staying (even) blocks per level
  DevBuf tabs, items, evens, binst, grp_lo, P, P2, E0, F0, F1, Rb, xp, hp;
  const int64_t* d_cols = nullptr;
  const int64_t* d_col0 = nullptr;
  const int64_t* d_row0 = nullptr;
  const int64_t* d_rows = nullptr;
  const int64_t* d_blk0 = nullptr;
  const int64_t* d_tail0 = nullptr;
};

static void release_splits(CRSplits* s) {
  for (DevBuf* b : {&s->item_blk, &s->blk_item0, &s->merges}) release(*b);
  delete s;
}

void release_cr(CRPlan*& p) {
  if (!p) return;
  for (CRSplits* s : p->splits) release_splits(s);
  for (DevBuf& b : p->outgrown) release(b);
  for (DevBuf* b : {&p->tabs, &p->items, &p->evens, &p->binst, &p->grp_lo, &p->P, &p->P2, &p->E0, &p->F0, &p->F1, &p->Rb,
                    &p->xp, &p->hp})
    release(*b);
  delete p;
  p = nullptr;
}

static qrkit_status upload(qrkit_ctx* ctx, DevBuf& d, const void* h, size_t bytes, const char* what) {
  qrkit_status r = ensure(ctx, d, std::max<size_t>(bytes, 8), what);
  if (r != QRKIT_OK) return r;
  if (bytes > 0) QRKIT_CUDA_TRY(ctx, cudaMemcpy(d.ptr, h, bytes, cudaMemcpyHostToDevice));
  return QRKIT_OK;
}

// A buffer of partial triangles of at least `parts`; an outgrown one is kept until the plan goes.  Each is at least twice
// the one before (or as large as there is room for), so that the kept ones together are no larger than the current.
static qrkit_status cr_partials(qrkit_ctx* ctx, CRPlan& C, DevBuf& buf, int64_t parts) {
  const size_t bytes = ((size_t)parts + 31) / 32 * 32 * kE0 * elem_size(ctx);
  if (parts == 0 || buf.bytes >= bytes) return QRKIT_OK;
  DevBuf grown;
  qrkit_status rc = QRKIT_ENOMEM;
  if (2 * buf.bytes > bytes) {
    rc = ensure(ctx, grown, 2 * buf.bytes, "banded partial triangles");
    if (rc == QRKIT_ENOMEM) cudaGetLastError();
  }
  if (rc != QRKIT_OK) rc = ensure(ctx, grown, bytes, "banded partial triangles");
  if (rc != QRKIT_OK) return rc;
  if (buf.ptr) C.outgrown.push_back(buf);
  buf = grown;
  return QRKIT_OK;
}

// The tables of a strategy: splits[k] threads per block of instance k.
static qrkit_status cr_split(qrkit_ctx* ctx, CRPlan& C, const std::vector<int>& splits, CRSplits& S) {
  for (int64_t k = 0; k < C.num_inst; ++k) S.num_items += (C.h_blk0[k + 1] - C.h_blk0[k]) * splits[k];
  if (S.num_items >= ((int64_t)1 << 31)) return fail(ctx, QRKIT_EUNSUPPORTED, "too many column blocks");
  if (S.num_items == C.total_blocks) return QRKIT_OK;   // one thread per block
  std::vector<int32_t> item_blk((size_t)S.num_items), item0((size_t)C.total_blocks + 1);
  std::vector<int32_t> first((size_t)C.total_blocks), n((size_t)C.total_blocks);   // a block's partials at this pass
  int64_t it = 0;
  for (int64_t k = 0; k < C.num_inst; ++k)
    for (int64_t gb = C.h_blk0[k]; gb < C.h_blk0[k + 1]; ++gb) {
      item0[gb] = first[gb] = (int32_t)it;
      n[gb] = splits[k];
      for (int q = 0; q < splits[k]; ++q) item_blk[it++] = (int32_t)gb;
    }
  item0[C.total_blocks] = (int32_t)it;
  std::vector<MergeItem> mg;
  int64_t parts2 = 0;
  for (bool more = true; more;) {
    more = false;
    S.mg_off.push_back((int64_t)mg.size());
    int64_t out = 0;
    for (int64_t gb = 0; gb < C.total_blocks; ++gb) {
      if (n[gb] <= 1) continue;
      const int m = (n[gb] + kMergeFan - 1) / kMergeFan;
      for (int q = 0; q < m; ++q)
        mg.push_back({(int32_t)gb, first[gb] + q * kMergeFan, std::min(kMergeFan, n[gb] - q * kMergeFan),
                      m == 1 ? -1 : (int32_t)(out + q)});
      first[gb] = (int32_t)out;
      n[gb] = m;
      if (m > 1) {
        out += m;
        more = true;
      }
    }
    parts2 = std::max(parts2, out);
    S.mg_n.push_back((int64_t)mg.size() - S.mg_off.back());
  }
  qrkit_status rc;
  if ((rc = upload(ctx, S.item_blk, item_blk.data(), item_blk.size() * 4, "banded splits")) != QRKIT_OK) return rc;
  if ((rc = upload(ctx, S.blk_item0, item0.data(), item0.size() * 4, "banded splits")) != QRKIT_OK) return rc;
  if ((rc = upload(ctx, S.merges, mg.data(), mg.size() * sizeof(MergeItem), "banded merges")) != QRKIT_OK) return rc;
  if ((rc = cr_partials(ctx, C, C.P, S.num_items)) != QRKIT_OK) return rc;
  return cr_partials(ctx, C, C.P2, parts2);
}

// Threads per block of each instance: about 800 per SM in all where that leaves each at least 64 rows (16 steps of four,
// what a merge pass takes), at most 64 per block.  A batch's instances differ in rows per block (curve fits: 60 to
// 10,000), and the longest thread bounds the kernel.  One LM step of 1,024 curve fits: 4,696 us at 400 per SM, 4,678 at
// 800, 4,711 at 1,600, 4,793 at 6,400; three steps of one curve fit of 200,000 points, which the rows bound: 1,570 us at
// least 32 rows, 1,397 at 64, 1,438 at 128.
// In double a thread takes about 10 us per row and a merge pass of up to four partials 320 us whatever is in it, so
// while the chip has room the powers of four are compared by rows per thread + 32 per pass (solve of 20,000 blocks 2 x 1
// with windows of 8 in 500 columns: 1,906 us at 64 rows per thread, 1,778; 300 columns of 40 rows: 1,813 and 1,620).
static std::vector<int> default_splits(const qrkit_ctx* ctx, const CRPlan& C) {
  std::vector<int> n((size_t)C.num_inst);
  const double target = std::max(64.0, (double)C.total_rows / (800.0 * ctx->num_sms));
  for (int64_t k = 0; k < C.num_inst; ++k) {
    const double per = (double)C.h_rows[k] / (double)(C.h_blk0[k + 1] - C.h_blk0[k]);
    if (elem_size(ctx) == 8) {
      const double least = (double)C.total_rows / (800.0 * ctx->num_sms);
      n[k] = 1;
      for (int m = 4, passes = 1; m <= 64 && per / m >= least; m *= 4, ++passes)
        if (per / m + 32.0 * passes < per / n[k] + 32.0 * (passes - 1)) n[k] = m;
        else break;
      continue;
    }
    n[k] = (int)std::min(64.0, std::max(1.0, std::floor(per / target + 0.5)));
  }
  return n;
}

// The current strategy becomes `each` threads per block, or (0) the default; on failure it stays what it was.
static qrkit_status cr_use_splits(qrkit_ctx* ctx, CRPlan& C, int each) {
  for (const CRSplits* s : C.splits)
    if (s->each == each) {
      C.cur = s;
      return QRKIT_OK;
    }
  const std::vector<int> n = each ? std::vector<int>((size_t)C.num_inst, each) : default_splits(ctx, C);
  CRSplits* s = new CRSplits();
  s->each = each;
  const qrkit_status rc = cr_split(ctx, C, n, *s);
  if (rc != QRKIT_OK) {
    release_splits(s);
    if (rc == QRKIT_ENOMEM) cudaGetLastError();   // reported; the next launch's check is not to find it
    return rc;
  }
  C.splits.push_back(s);
  C.cur = s;
  return QRKIT_OK;
}

qrkit_status cr_build(qrkit_ctx* ctx, CRPlan*& out, const std::vector<int64_t>& cols,
                      const std::vector<int64_t>& col0, const std::vector<int64_t>& row0,
                      const std::vector<int64_t>& rows) {
  release_cr(out);
  out = new CRPlan();
  CRPlan& C = *out;
  const int64_t ni = (int64_t)cols.size();
  C.num_inst = ni;
  std::vector<int64_t> blk0(ni + 1, 0);
  for (int64_t k = 0; k < ni; ++k) {
    if (cols[k] < 1) return fail(ctx, QRKIT_EINVAL, "banded instance without columns");
    blk0[k + 1] = blk0[k] + (cols[k] + kCB - 1) / kCB;
    C.total_rows += rows[k];
  }
  C.total_blocks = blk0[ni];
  if (C.total_blocks >= ((int64_t)1 << 30)) return fail(ctx, QRKIT_EUNSUPPORTED, "too many column blocks");
  C.h_blk0 = blk0;
  C.h_rows = rows;
  // level work lists; an instance's levels with at most kTailBlocks blocks belong to its tail
  std::vector<std::vector<int64_t>> lv, ev;
  std::vector<int64_t> tail0(ni);
  for (int64_t k = 0; k < ni; ++k) {
    int64_t Gl = blk0[k + 1] - blk0[k];
    int l = 0;
    for (; Gl > kTailBlocks; ++l) {
      if ((int)lv.size() <= l) {
        lv.emplace_back();
        ev.emplace_back();
      }
      for (int64_t i = 1; i < Gl; i += 2) lv[l].push_back((k << 32) | (i << 2) | 0);
      if (Gl % 2 == 1) lv[l].push_back((k << 32) | ((Gl - 1) << 2) | 1);
      for (int64_t j = 0; j < Gl; j += 2) ev[l].push_back((k << 32) | j);
      Gl = (Gl + 1) / 2;
    }
    tail0[k] = l;
  }
  C.levels = (int)lv.size();
  std::vector<int64_t> items, evens;
  for (int l = 0; l < C.levels; ++l) {
    C.lvl_off.push_back((int64_t)items.size());
    C.lvl_n.push_back((int64_t)lv[l].size());
    items.insert(items.end(), lv[l].begin(), lv[l].end());
    C.ev_off.push_back((int64_t)evens.size());
    C.ev_n.push_back((int64_t)ev[l].size());
    evens.insert(evens.end(), ev[l].begin(), ev[l].end());
  }
  std::vector<int64_t> tabs;
  for (const auto* v : {&cols, &col0, &row0, &rows}) tabs.insert(tabs.end(), v->begin(), v->end());
  tabs.insert(tabs.end(), blk0.begin(), blk0.end());
  tabs.insert(tabs.end(), tail0.begin(), tail0.end());
  std::vector<int32_t> binst((size_t)C.total_blocks);
  for (int64_t k = 0; k < ni; ++k) std::fill(binst.begin() + blk0[k], binst.begin() + blk0[k + 1], (int32_t)k);
  qrkit_status rc;
  if ((rc = upload(ctx, C.tabs, tabs.data(), tabs.size() * sizeof(int64_t), "banded tables")) != QRKIT_OK) return rc;
  if ((rc = upload(ctx, C.items, items.data(), items.size() * sizeof(int64_t), "banded levels")) != QRKIT_OK) return rc;
  if ((rc = upload(ctx, C.evens, evens.data(), evens.size() * sizeof(int64_t), "banded levels")) != QRKIT_OK) return rc;
  if ((rc = upload(ctx, C.binst, binst.data(), binst.size() * sizeof(int32_t), "banded blocks")) != QRKIT_OK) return rc;
  const int64_t* t = (const int64_t*)C.tabs.ptr;
  C.d_cols = t;
  C.d_col0 = t + ni;
  C.d_row0 = t + 2 * ni;
  C.d_rows = t + 3 * ni;
  C.d_blk0 = t + 4 * ni;
  C.d_tail0 = t + 5 * ni + 1;
  const size_t es = elem_size(ctx);
  const size_t TB = (size_t)C.total_blocks;
  if ((rc = ensure(ctx, C.grp_lo, TB * sizeof(int64_t), "banded group rows")) != QRKIT_OK) return rc;
  if ((rc = cr_use_splits(ctx, C, 0)) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.E0, (TB + 31) / 32 * 32 * kE0 * es, "banded block rows")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.F0, TB * kFW * es, "banded block rows")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.F1, TB * kFW * es, "banded block rows")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.Rb, TB * kRW * es, "banded R blocks")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.xp, TB * kCB * es, "banded padded x")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.hp, TB * kCB * es, "banded padded h")) != QRKIT_OK) return rc;
  return QRKIT_OK;
}

qrkit_status cr_set_strategy(qrkit_ctx* ctx, CRPlan& C, int splits) {
  if (splits < 0 || splits > 64) return fail(ctx, QRKIT_EINVAL, "splits must be in [1, 64]");
  return cr_use_splits(ctx, C, splits);
}

std::vector<int> cr_candidates(const qrkit_ctx* ctx, const CRPlan& C) {
  const std::vector<int> def = default_splits(ctx, C);
  const bool uniform = std::all_of(def.begin(), def.end(), [&](int n) { return n == def[0]; });
  double most = 0.0;   // rows per block
  for (int64_t k = 0; k < C.num_inst; ++k)
    most = std::max(most, (double)C.h_rows[k] / (double)(C.h_blk0[k + 1] - C.h_blk0[k]));
  std::vector<int> c{0};
  for (const int n : {1, 2, 4, 8, 16, 32, 64})
    if ((n <= 8 || 4 * n <= most) && !(uniform && n == def[0])) c.push_back(n);   // a step is four rows
  return c;
}

CRTuning cr_tuning_begin(const CRPlan& C) { return {C.splits.size(), C.outgrown.size(), C.P.ptr, C.P2.ptr}; }

void cr_tuning_end(CRPlan& C, const CRTuning& before) {
  // the timing has ended, and nothing else has been told of what it built
  for (size_t q = before.strategies; q < C.splits.size();) {
    if (C.splits[q] == C.cur) {
      ++q;
    } else {
      release_splits(C.splits[q]);
      C.splits.erase(C.splits.begin() + (int64_t)q);
    }
  }
  for (size_t q = before.outgrown; q < C.outgrown.size();) {
    if (C.outgrown[q].ptr == before.P || C.outgrown[q].ptr == before.P2) {
      ++q;
    } else {
      release(C.outgrown[q]);
      C.outgrown.erase(C.outgrown.begin() + (int64_t)q);
    }
  }
}

template <typename T>
static CRArgs<T> cr_args(qrkit_ctx* ctx, CRPlan& C) {
  CRArgs<T> A{};
  A.num_inst = C.num_inst;
  A.cols = C.d_cols;
  A.col0 = C.d_col0;
  A.row0 = C.d_row0;
  A.rows = C.d_rows;
  A.blk0 = C.d_blk0;
  A.tail0 = C.d_tail0;
  A.binst = (const int32_t*)C.binst.ptr;
  A.total_blocks = C.total_blocks;
  A.num_items = C.cur->num_items;
  A.item_blk = (const int32_t*)C.cur->item_blk.ptr;   // both null for one thread per block
  A.blk_item0 = (const int32_t*)C.cur->blk_item0.ptr;
  A.grp_lo = (int64_t*)C.grp_lo.ptr;
  A.P = (T*)C.P.ptr;
  A.E0 = (T*)C.E0.ptr;
  A.F0 = (T*)C.F0.ptr;
  A.F1 = (T*)C.F1.ptr;
  A.Rb = (T*)C.Rb.ptr;
  A.xp = (T*)C.xp.ptr;
  A.hp = (T*)C.hp.ptr;
  A.status = ctx->d_status;
  return A;
}

// CR_LAUNCH(ctx, grid, block, shared memory, kernel, arguments ..)
#define CR_LAUNCH(ctx, ...)                                      \
  do {                                                           \
    QRKIT_CUDA_TRY(ctx, chain_launch((ctx)->stream, __VA_ARGS__)); \
    (ctx)->launches += 1;                                        \
  } while (0)

template <typename T>
static qrkit_status cr_solve_typed(qrkit_ctx* ctx, CRPlan& C, const int64_t* starts, const int32_t* colptr, int rpc, int w,
                                   const T* J, const T* b, const double* D, double lambda, T* x, double* res2) {
  cudaStream_t st = ctx->stream;
  CRArgs<T> A = cr_args<T>(ctx, C);
  A.starts = starts;
  A.colptr = colptr;
  A.rpc = rpc;
  A.w = w;
  A.J = J;
  A.b = b;
  A.D = D;
  A.lam = lambda;
  A.res2 = res2;
  QRKIT_CUDA_TRY(ctx, cudaMemsetAsync(res2, 0, (size_t)C.num_inst * sizeof(double), st));
  if (starts) CR_LAUNCH(ctx, nblk(C.total_blocks, 256), 256, 0, cr_ranges_kernel<T>, A);
  const CRSplits& S = *C.cur;
  const unsigned cgrid = nblk(S.num_items, kCompThreads);
  if (w == kCB && (reinterpret_cast<uintptr_t>(J) & 15) == 0) {
    const size_t smem = 2 * (size_t)kCompThreads * stage_stride<T>();
    auto kc = cr_compress_kernel<T, true>;
    if (smem > 48 * 1024)
      QRKIT_CUDA_TRY(ctx, cudaFuncSetAttribute(kc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    CR_LAUNCH(ctx, cgrid, kCompThreads, smem, kc, A);
  } else {
    CR_LAUNCH(ctx, cgrid, kCompThreads, 0, (cr_compress_kernel<T, false>), A);
  }
  T* in = A.P;
  T* other = (T*)C.P2.ptr;
  for (size_t q = 0; q < S.mg_n.size(); ++q) {
    CR_LAUNCH(ctx, nblk(S.mg_n[q], kCompThreads), kCompThreads, 0, cr_merge_kernel<T>, A,
              (const MergeItem*)S.merges.ptr + S.mg_off[q], S.mg_n[q], in, other);
    std::swap(in, other);
  }
  const int64_t* items = (const int64_t*)C.items.ptr;
  for (int l = 0; l < C.levels; ++l) {
    const T* Fc = l == 0 ? A.E0 : ((l & 1) ? A.F1 : A.F0);
    T* Fn = (l & 1) ? A.F0 : A.F1;
    const unsigned grid = nblk(C.lvl_n[l] * kItemThreads, kLevelThreads);
    if (l == 0)
      CR_LAUNCH(ctx, grid, kLevelThreads, 0, (cr_level_kernel<T, true>), A, items + C.lvl_off[l],
                C.lvl_n[l], l, Fc, Fn);
    else
      CR_LAUNCH(ctx, grid, kLevelThreads, 0, (cr_level_kernel<T, false>), A, items + C.lvl_off[l],
                C.lvl_n[l], l, Fc, Fn);
  }
  const int tt = C.num_inst >= 4 * ctx->num_sms ? 128 : tail_threads<T>();
  CR_LAUNCH(ctx, (unsigned)C.num_inst, tt, 0, cr_tail_kernel<T>, A, x);
  for (int l = C.levels - 1; l >= 0; --l)
    CR_LAUNCH(ctx, nblk(C.lvl_n[l] * kItemThreads, 128), 128, 0, cr_backsub_kernel<T>, A, items + C.lvl_off[l],
              C.lvl_n[l], l, 0, x, (T*)nullptr);
  return QRKIT_OK;
}

// dx = R^{-1} R^{-T} g with the stored factor (g: double over global columns, or null: already in the
// padded layout), written to dx and added to xadd (either may be null).
template <typename T>
static qrkit_status cr_normal_typed(qrkit_ctx* ctx, CRPlan& C, const double* g, T* dx, T* xadd) {
  CRArgs<T> A = cr_args<T>(ctx, C);
  const int64_t* items = (const int64_t*)C.items.ptr;
  const int64_t* evens = (const int64_t*)C.evens.ptr;
  if (g) CR_LAUNCH(ctx, nblk(C.total_blocks * kCB, 256), 256, 0, cr_scatter_g_kernel<T>, A, g);
  for (int l = 0; l < C.levels; ++l)
    CR_LAUNCH(ctx, nblk(C.ev_n[l] * kItemThreads, 128), 128, 0, cr_rt_level_kernel<T>, A, evens + C.ev_off[l],
              C.ev_n[l], l);
  const int tt = C.num_inst >= 4 * ctx->num_sms ? 128 : tail_threads<T>();
  CR_LAUNCH(ctx, (unsigned)C.num_inst, tt, 0, cr_tail_normal_kernel<T>, A, dx, xadd);
  for (int l = C.levels - 1; l >= 0; --l)
    CR_LAUNCH(ctx, nblk(C.lvl_n[l] * kItemThreads, 128), 128, 0, cr_backsub_kernel<T>, A, items + C.lvl_off[l],
              C.lvl_n[l], l, 1, dx, xadd);
  return QRKIT_OK;
}

void cr_padded(const CRPlan& C, const int64_t** blk0, void** g) {
  *blk0 = C.d_blk0;
  *g = C.xp.ptr;
}

qrkit_status cr_solve(qrkit_ctx* ctx, CRPlan& C, const int64_t* starts, const int32_t* colptr, int rpc, int w,
                      const void* J, const void* b, const double* D, double lambda, void* x, double* res2) {
  if (w < 1 || w > kCB) return fail(ctx, QRKIT_EUNSUPPORTED, "the parallel banded QR needs w <= 8");
  if (ctx->precision == QRKIT_FP64)
    return cr_solve_typed<double>(ctx, C, starts, colptr, rpc, w, (const double*)J, (const double*)b, D, lambda,
                                  (double*)x, res2);
  return cr_solve_typed<float>(ctx, C, starts, colptr, rpc, w, (const float*)J, (const float*)b, D, lambda, (float*)x,
                               res2);
}

qrkit_status cr_normal_solve(qrkit_ctx* ctx, CRPlan& C, const double* g, void* dx, void* xadd) {
  if (ctx->precision == QRKIT_FP64) return cr_normal_typed<double>(ctx, C, g, (double*)dx, (double*)xadd);
  return cr_normal_typed<float>(ctx, C, g, (float*)dx, (float*)xadd);
}

}  // namespace qrkit
