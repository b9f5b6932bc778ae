// Block-banded QR of P_r [J; lambda^(1/2) D] (Sec. 4.4 "Block banded", Sec. 4.5 / Sec. 5.2
// row interleave of the damping rows) and the banded solve, for batches of independent
// banded instances.
//
// J row i of an instance touches columns floor(i / rows_per_col) .. + w - 1 (entries past the
// last column are ignored); values are stored row-major, w per row.  The damping row of
// column j has the single value lambda^(1/2) D_j at column j.
//
// Work mapping: one warp per instance, several instances per CTA.  The warp sweeps column
// groups [c0, c0 + 8): the front holds the rows carried from the previous group (at most
// w - 1, non-zero only from column c0 on) plus the J rows and damping rows whose first column
// lies in the group; rows are appended in batches to a shared-memory front and reduced by
// Householder reflections (Sec. 2) with lanes over columns, so the front never holds more
// than (group + w - 1) + batch rows however dense the rows are.  After the last batch the
// group's R rows are final (written as windows R[j, j .. j + w - 1]) and the next w - 1 rows
// are carried.  Every Householder vector is as long as its front, never as long as the
// matrix (Sec. 4.4).  Q is not kept: the right-hand side is reflected along with the front.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "chain.cuh"
#include "device_util.cuh"
#include "f32x2.cuh"
#include "internal.h"
#include "sums.cuh"

namespace qrkit {
namespace {

constexpr int kBG = 8;          // columns per group
constexpr int kBW = 16;         // largest band window
constexpr int kBatch = 48;      // new rows appended per front reduction
constexpr int kFCols = kBG + kBW - 1 + 1;      // front columns incl. the rhs column
constexpr int kFStride = kFCols + 1;           // padded row stride (bank spread)
constexpr int kFRows = kBG + kBW - 1 + kBatch; // kept rows + one batch
constexpr int kWarps = 4;                      // instances per CTA (float)
template <typename T> constexpr int warps_for() { return sizeof(T) == sizeof(double) ? 2 : kWarps; }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

__device__ __forceinline__ void brecord(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

template <typename T>
struct BandArgs {
  int64_t num_inst;
  const int64_t* inst_cols;   // columns per instance
  const int64_t* inst_col0;   // first global column of each instance
  const int64_t* inst_row0;   // first J row of each instance
  int rows_per_col;           // implicit row starts: row i starts at floor(i / rows_per_col)
  const int64_t* row_start;   // explicit row starts, global columns, non-decreasing per instance (null: implicit)
  const int64_t* inst_rows;   // rows per instance when row_start is given
  int w;                      // band window (<= kBW)
  const T* J;                 // rows x w, row-major
  const T* b;                 // rows
  const double* D;            // global columns (may be null when !damp)
  double lam;                 // lambda (damping rows present iff lam > 0)
  T* Rw;                      // global columns x w: R[j, j + t] at Rw[j * w + t]
  T* c;                       // global columns: top of Q^T [b; 0]
  T* x;                       // global columns: solution
  double* res2;               // per instance: squared norm of the rest of Q^T [b; 0]
  int refine_steps;
  int* status;
};

// One reduction of the front F (nr rows x fc columns + rhs column fc) by Householder
// reflections, column by column; lanes over columns for the dot products and updates.
template <typename T>
__device__ __forceinline__ void front_qr(T* F, int nr, int fc, int lane) {
  const int kmax = nr < fc ? nr : fc;
  for (int k = 0; k < kmax; ++k) {
    T s = 0;
    for (int r = k + 1 + lane; r < nr; r += 32) {
      const T a = F[r * kFStride + k];
      s += a * a;
    }
    s = warp_sum(s);
    const T alpha = F[k * kFStride + k];
    const T norm = sqrt(alpha * alpha + s);
    T beta = 0, tau = 0, scale = 0;
    if (norm != T(0)) {
      beta = alpha >= T(0) ? -norm : norm;
      tau = (beta - alpha) / beta;
      scale = T(1) / (alpha - beta);
    }
    for (int r = k + 1 + lane; r < nr; r += 32) F[r * kFStride + k] *= scale;
    __syncwarp();
    const int j = k + 1 + lane;   // one lane per trailing column (incl. the rhs column fc)
    if (j <= fc) {
      T wv = F[k * kFStride + j];
      for (int r = k + 1; r < nr; ++r) wv += F[r * kFStride + k] * F[r * kFStride + j];
      wv *= tau;
      F[k * kFStride + j] -= wv;
      for (int r = k + 1; r < nr; ++r) F[r * kFStride + j] -= wv * F[r * kFStride + k];
    }
    __syncwarp();
    if (lane == 0) F[k * kFStride + k] = beta;
    for (int r = k + 1 + lane; r < nr; r += 32) F[r * kFStride + k] = T(0);
    __syncwarp();
  }
}

template <typename T>
__global__ void __launch_bounds__(32 * kWarps)
banded_factor_solve_kernel(BandArgs<T> A) {
  constexpr int NW = warps_for<T>();   // static shared memory stays under 48 KB
  __shared__ __align__(16) T sF[NW][kFRows * kFStride];
  const int lane = threadIdx.x & 31;
  const int wid = threadIdx.x >> 5;
  const int64_t inst = (int64_t)blockIdx.x * NW + wid;
  if (inst >= A.num_inst) return;
  T* F = sF[wid];
  const int w = A.w;
  const int64_t N = A.inst_cols[inst];
  const int64_t col0 = A.inst_col0[inst];
  const int64_t row0 = A.inst_row0[inst];
  const int64_t nrows = A.row_start ? A.inst_rows[inst] : (int64_t)A.rows_per_col * N;
  const bool damp = A.lam > 0.0;
  const double lam_half = sqrt(A.lam);
  double res2 = 0.0;
  int carried = 0;   // rows 0 .. carried-1 of F hold the carried rows (columns from c0 on)
  int64_t jr_next = 0;   // explicit starts: first row not yet consumed
  for (int e = lane; e < kFRows * kFStride; e += 32) F[e] = T(0);
  __syncwarp();
  for (int64_t c0 = 0; c0 < N; c0 += kBG) {
    const int64_t c1 = c0 + kBG < N ? c0 + kBG : N;
    const int g = (int)(c1 - c0);
    const int64_t hi = c1 + w - 1 < N ? c1 + w - 1 : N;
    const int fc = (int)(hi - c0);            // front columns; the rhs sits in column fc
    // the rhs column index changes with fc: move the carried rows' rhs into place
    // (carried rows were written with the rhs at column kFCols - 1, see below)
    for (int r = lane; r < carried; r += 32) {
      const T rhs = F[r * kFStride + (kFCols - 1)];
      F[r * kFStride + (kFCols - 1)] = T(0);
      F[r * kFStride + fc] = rhs;
    }
    __syncwarp();
    int nr = carried;
    // stream of new rows: J rows starting in [c0, c1), then the damping rows of c0 .. c1-1
    int64_t jr, jr_end;
    if (A.row_start) {
      jr = jr_next;
      jr_end = jr;
      while (jr_end < nrows && A.row_start[row0 + jr_end] - col0 < c1) ++jr_end;
      jr_next = jr_end;
    } else {
      jr = (int64_t)A.rows_per_col * c0;
      jr_end = (int64_t)A.rows_per_col * c1 < nrows ? (int64_t)A.rows_per_col * c1 : nrows;
    }
    int64_t dr = damp ? c0 : c1;
    while (jr < jr_end || dr < c1) {
      const int room = kFRows - nr;
      const int64_t take_j = jr_end - jr < room ? jr_end - jr : room;
      const int64_t take_d = (c1 - dr) < (room - take_j) ? (c1 - dr) : (room - take_j);
      // append (lanes over new rows); each row is cleared first
      for (int t = lane; t < (int)(take_j + take_d); t += 32) {
        T* row = F + (nr + t) * kFStride;
        for (int q = 0; q < kFStride; ++q) row[q] = T(0);
        if (t < take_j) {
          const int64_t i = jr + t;
          const int64_t start = A.row_start ? A.row_start[row0 + i] - col0 : i / A.rows_per_col;
          const T* src = A.J + (row0 + i) * w;
          for (int q = 0; q < w; ++q) {
            const int64_t col = start + q;
            if (col >= c0 && col < N) row[col - c0] = src[q];
          }
          row[fc] = A.b[row0 + i];
        } else {
          const int64_t j = dr + (t - take_j);
          row[j - c0] = (T)(lam_half * A.D[col0 + j]);
        }
      }
      __syncwarp();
      nr += (int)(take_j + take_d);
      jr += take_j;
      dr += take_d;
      front_qr(F, nr, fc, lane);
      // rows beyond the triangle are now zero: their rhs is residual
      double part = 0.0;
      for (int r = fc + lane; r < nr; r += 32) {
        const double v = (double)F[r * kFStride + fc];
        part += v * v;
        F[r * kFStride + fc] = T(0);
      }
      res2 += warp_sum(part);
      nr = nr < fc ? nr : fc;
      __syncwarp();
    }
    if (nr < g) {
      brecord(A.status, QRKIT_ESINGULAR);   // fewer rows than columns in this group
    }
    // final R rows of the group
    for (int i = lane; i < g; i += 32) {
      const int64_t gj = col0 + c0 + i;
      for (int t = 0; t < w; ++t) {
        const int colf = i + t;
        A.Rw[gj * w + t] = (colf < fc && i < nr) ? F[i * kFStride + colf] : T(0);
      }
      A.c[gj] = i < nr ? F[i * kFStride + fc] : T(0);
    }
    __syncwarp();
    // carry rows g .. nr-1, shifted left by g columns; rhs parked in column kFCols - 1
    const int nc = nr - g > 0 ? nr - g : 0;
    if (c1 < N) {
      // ascending rows: the source row g + r is read before any later row overwrites it
      for (int r = 0; r < nc; ++r) {
        const T* src = F + (g + r) * kFStride;
        T v = T(0);
        if (lane < kFCols - 1 && lane + g < fc) v = src[lane + g];
        const T rhs = src[fc];
        __syncwarp();
        T* dst = F + r * kFStride;
        if (lane < kFCols - 1) dst[lane] = v;
        if (lane == 0) dst[kFCols - 1] = rhs;
        __syncwarp();
      }
      // clear the rows above the carried ones
      for (int e = nc * kFStride + lane; e < kFRows * kFStride; e += 32) F[e] = T(0);
      __syncwarp();
    }
    carried = nc;
  }
  if (lane == 0) A.res2[inst] = res2;
  // back-substitution R x = c on the banded R (one lane; the recurrence is sequential)
  if (lane == 0) {
    bool bad = false;
    for (int64_t j = N - 1; j >= 0; --j) {
      const int64_t gj = col0 + j;
      T s = A.c[gj];
      for (int t = 1; t < w && j + t < N; ++t) s -= A.Rw[gj * w + t] * A.x[gj + t];
      const T rjj = A.Rw[gj * w];
      if (rjj == T(0)) bad = true;
      A.x[gj] = s / rjj;
    }
    if (bad) brecord(A.status, QRKIT_ESINGULAR);
  }
}

// ---- refinement for float instances: r = b - J x in double (one lane per row), then
// g = J^T r - lambda D^2 x (one lane per column), then x += R^{-1} R^{-T} g by banded
// triangular solves; one warp per instance ----
__global__ void __launch_bounds__(32 * kWarps)
banded_refine_kernel(BandArgs<float> A, double* rbuf, double* gbuf, float* hbuf) {
  const int lane = threadIdx.x & 31;
  const int wid = threadIdx.x >> 5;
  const int64_t inst = (int64_t)blockIdx.x * kWarps + wid;
  if (inst >= A.num_inst) return;
  const int w = A.w;
  const int rpc = A.rows_per_col;
  const int64_t N = A.inst_cols[inst];
  const int64_t col0 = A.inst_col0[inst];
  const int64_t row0 = A.inst_row0[inst];
  const int64_t nrows = (int64_t)rpc * N;
  for (int64_t i = lane; i < nrows; i += 32) {
    const int64_t s = i / rpc;
    const float* row = A.J + (row0 + i) * w;
    double r = (double)A.b[row0 + i];
    for (int t = 0; t < w && s + t < N; ++t) r -= (double)row[t] * (double)A.x[col0 + s + t];
    rbuf[row0 + i] = r;
  }
  __syncwarp();
  for (int64_t j = lane; j < N; j += 32) {
    double acc = 0.0;
    const int64_t s_lo = j - w + 1 > 0 ? j - w + 1 : 0;
    for (int64_t s = s_lo; s <= j; ++s)
      for (int q = 0; q < rpc; ++q) {
        const int64_t i = s * rpc + q;
        if (i >= nrows) break;
        acc += (double)A.J[(row0 + i) * w + (j - s)] * rbuf[row0 + i];
      }
    if (A.lam > 0.0) {
      const double d = A.D[col0 + j];
      acc -= A.lam * d * d * (double)A.x[col0 + j];
    }
    gbuf[col0 + j] = acc;
  }
  __syncwarp();
  if (lane == 0) {
    // R^T h = g (forward): h_j = (g_j - sum_{t=1}^{w-1} R[j-t, j] h_{j-t}) / R[j, j]
    for (int64_t j = 0; j < N; ++j) {
      const int64_t gj = col0 + j;
      float s = (float)gbuf[gj];
      for (int t = 1; t < w && j - t >= 0; ++t) s -= A.Rw[(gj - t) * w + t] * hbuf[gj - t];
      hbuf[gj] = s / A.Rw[gj * w];
    }
    // R dx = h (backward), x += dx
    for (int64_t j = N - 1; j >= 0; --j) {
      const int64_t gj = col0 + j;
      float s = hbuf[gj];
      for (int t = 1; t < w && j + t < N; ++t) s -= A.Rw[gj * w + t] * hbuf[gj + t];
      hbuf[gj] = s / A.Rw[gj * w];
    }
    for (int64_t j = 0; j < N; ++j) A.x[col0 + j] += hbuf[col0 + j];
  }
}

// R^T h = g (transpose = 1: forward with R^T) or R x = h (backward) for the banded R of each
// instance (windows Rw by global column); one thread per instance, the recurrences are
// sequential.  In place on v (global columns).
template <typename T>
__global__ void band_tri_solve_kernel(int64_t num_inst, const int64_t* inst, const T* Rw, int w, T* v,
                                      int transpose) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= num_inst) return;
  const int64_t n = inst[k], c0 = inst[num_inst + k];
  const T* R = Rw + c0 * w;
  T* x = v + c0;
  if (transpose) {
    for (int64_t j = 0; j < n; ++j) {
      T s = x[j];
      for (int t = 1; t < w && j - t >= 0; ++t) s -= R[(j - t) * w + t] * x[j - t];
      x[j] = s / R[j * w];
    }
  } else {
    for (int64_t j = n - 1; j >= 0; --j) {
      T s = x[j];
      for (int t = 1; t < w && j + t < n; ++t) s -= R[j * w + t] * x[j + t];
      x[j] = s / R[j * w];
    }
  }
}

__global__ void band_colnorm_kernel(const float* Jf, const double* Jd, const int64_t* inst_cols,
                                    const int64_t* inst_col0, const int64_t* inst_row0,
                                    int64_t num_inst, int rpc, int w, double* D) {
  // one thread per global column: rows touching column j start in [j - w + 1, j]
  const int64_t total = inst_col0[num_inst - 1] + inst_cols[num_inst - 1];
  const int64_t gj = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (gj >= total) return;
  int64_t lo = 0, hi = num_inst - 1;
  while (lo < hi) {   // instance of column gj
    const int64_t mid = (lo + hi + 1) / 2;
    if (inst_col0[mid] <= gj) lo = mid; else hi = mid - 1;
  }
  const int64_t inst = lo, j = gj - inst_col0[inst], N = inst_cols[inst];
  const int64_t nrows = (int64_t)rpc * N;
  double acc = 0.0;
  const int64_t s_lo = j - w + 1 > 0 ? j - w + 1 : 0;
  for (int64_t s = s_lo; s <= j; ++s)
    for (int q = 0; q < rpc; ++q) {
      const int64_t i = s * rpc + q;
      if (i >= nrows) break;
      const int64_t e = (inst_row0[inst] + i) * w + (j - s);
      const double v = Jf ? (double)Jf[e] : Jd[e];
      acc += v * v;
    }
  const double d = sqrt(acc);
  D[gj] = d == 0.0 ? 1.0 : d;
}

// Float J with implicit row starts: the column norms and the refinement gradient, by row groups.
// Group c (column c of the concatenated instances) holds the rpc rows that start at column c, so column j's
// entries are entry t of groups j - t, t < w.  A CTA of NT threads takes NT consecutive groups, of which the last
// NT - (w - 1) are its columns: their rows arrive in shared memory by coalesced 16-byte cp.async copies (a
// thread reading its own group from global memory touches a cache line of its own at every load), thread t
// computes the sums of group t per diagonal, and then the column of group t from the w sums on its anti-diagonal.
// The rows' residuals are formed on the way, so a refinement step reads J once.
// 256 instances, 13 million columns, 4 rows of 8 values per column (1.87 GB): 344 us for the norms
// (2 phases reading global memory 1,000), 633 us per gradient (residual 636 and gradient 1,738; 728 with
// scalar sums), bound by the additions of the pair sums.
template <bool kStaged>
__device__ __forceinline__ const float* group_rows_f32(const float* J, int64_t grp0, int64_t total, int rw, int gs,
                                                       float* buf) {
  const int nt = blockDim.x;
  if constexpr (kStaged) {
    const bool wide = (rw & 3) == 0 && (reinterpret_cast<uintptr_t>(J) & 15) == 0;   // then gs % 4 == 0 too
    const int unit = wide ? 4 : 1, per = rw / unit;
    int gg = threadIdx.x / per, o = (threadIdx.x - gg * per) * unit;   // of the thread's next copy
    const int dg = nt / per, dq = (nt - dg * per) * unit;
    const float* src0 = J + grp0 * rw;
    const int lo = grp0 < 0 ? (int)-grp0 : 0, hi = (int)(total - grp0 < nt ? total - grp0 : nt);
    for (int e = 0; e < per; ++e) {
      if (gg >= lo && gg < hi) {
        const float* src = src0 + gg * rw + o;
        float* dst = buf + gg * gs + o;
        if (wide) dev::cp_async16(dst, src);
        else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dev::smem_u32(dst)), "l"(src) : "memory");
      }
      gg += dg;
      o += dq;
      if (o >= rw) {
        o -= rw;
        ++gg;
      }
    }
    dev::cp_async_commit();
    dev::cp_async_wait_all();
    return buf + threadIdx.x * gs;
  } else {
    return J + (grp0 + threadIdx.x) * (int64_t)rw;
  }
}

// Instance of group grp: from the CTA's first instance onwards.
__device__ __forceinline__ int64_t instance_of_group(const int64_t* inst_col0, const int64_t* inst_cols,
                                                     int64_t num_inst, int64_t grp0, int64_t grp) {
  __shared__ int64_t first;
  if (threadIdx.x == 0) {
    int64_t lo = 0, hi = num_inst - 1;
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) / 2;
      if (inst_col0[mid] <= (grp0 > 0 ? grp0 : 0)) lo = mid; else hi = mid - 1;
    }
    first = lo;
  }
  __syncthreads();
  int64_t k = first;
  while (k + 1 < num_inst && inst_col0[k] + inst_cols[k] <= grp) ++k;
  return k;
}

// A row's w values (a fixed 8 by two 16-byte loads, or any w <= MW).
template <bool kW8, int MW>
__device__ __forceinline__ void row_f32(float (&a)[MW], const float* row, int w) {
  if constexpr (kW8) {
    const float4 p = reinterpret_cast<const float4*>(row)[0], q = reinterpret_cast<const float4*>(row)[1];
    a[0] = p.x; a[1] = p.y; a[2] = p.z; a[3] = p.w;
    a[4] = q.x; a[5] = q.y; a[6] = q.z; a[7] = q.w;
  } else {
#pragma unroll
    for (int t = 0; t < MW; ++t) a[t] = t < w ? row[t] : 0.f;
  }
}

struct BandGroups {   // what both kernels are told
  const float* J;
  int64_t total_cols;
  const int64_t* inst_cols;
  const int64_t* inst_col0;
  int64_t num_inst;
  int rpc, w, gs;   // gs: stride of a staged group
};

// lambda D^2 of a column as a float pair, for the gradient: float arithmetic while lambda and D^2 are of a size whose
// products stay exact, double otherwise (a given D may balance a lambda of any size).
struct BandDamping {
  double lam;
  float h, l;       // lambda as a pair
  bool ordinary;    // 2^-60 <= lambda <= 2^60
  explicit BandDamping(double x)
      : lam(x), h((float)x), l((float)(x - (double)(float)x)), ordinary(x >= 0x1p-60 && x <= 0x1p60) {}
  // times D^2 = s + e; dd: D^2 in double
  template <class F>
  __device__ __forceinline__ float2 times(float s, float e, F&& dd) const {
    if (ordinary && s >= 0x1p-40f && s <= 0x1p60f) {
      const float p = __fmul_rn(h, s);
      return make_float2(p, __fmaf_rn(h, e, __fmaf_rn(l, s, __fmaf_rn(h, s, -p))));
    }
    const double v = lam * dd();
    return make_float2((float)v, (float)(v - (double)(float)v));
  }
};

// The group sums are floats, as accurate as the entries' squares; what follows them is done in float pairs and adds
// nothing to their error.
template <bool kW8, bool kStaged, int MW>
__global__ void __launch_bounds__(256) band_norm_f32_kernel(BandGroups B, BandDamping damp, double* D, float2* E2) {
  dev::chain_wait();
  extern __shared__ __align__(16) float sm_f[];
  const int nt = blockDim.x, tid = threadIdx.x, w = B.w;
  const int64_t grp0 = (int64_t)blockIdx.x * (nt - (w - 1)) - (w - 1), grp = grp0 + tid;
  const float* rows = group_rows_f32<kStaged>(B.J, grp0, B.total_cols, B.rpc * w, B.gs, sm_f);
  float* S = sm_f + (kStaged ? nt * B.gs : 0);   // per group and diagonal, stride w + 1
  const int64_t k = instance_of_group(B.inst_col0, B.inst_cols, B.num_inst, grp0, grp);   // and the staged rows
  const bool have = grp >= 0 && grp < B.total_cols;
  float acc[MW];
#pragma unroll
  for (int t = 0; t < MW; ++t) acc[t] = 0.f;
  if (have)
    for (int q = 0; q < B.rpc; ++q) {
      float a[MW];
      row_f32<kW8, MW>(a, rows + (int64_t)q * w, w);
#pragma unroll
      for (int t = 0; t < MW; ++t) acc[t] += a[t] * a[t];
    }
#pragma unroll
  for (int t = 0; t < MW; ++t)
    if (t < w) S[tid * (w + 1) + t] = acc[t];
  __syncthreads();
  if (tid < w - 1 || !have) return;
  const int64_t j = grp - B.inst_col0[k];
  float h = 0.f, l = 0.f;   // the sum, and then its root, as float pairs
  for (int t = 0; t < w && t <= j; ++t) dev::pair_add(h, l, S[(tid - t) * (w + 1) + t], 0.f);
  const float s = h + l;
  l = (h - s) + l;
  float r = s, c = 0.f;   // NaN and infinity are their own root
  if (s > 0.f && s <= 3.4e38f) {
    r = sqrtf(s);
    c = (__fmaf_rn(-r, r, s) + l) / (2.f * r);   // one Newton step for the root of s + l
  } else if (s == 0.f) {   // zero norm -> 1
    E2[grp] = damp.times(1.f, 0.f, [] { return 1.0; });
    D[grp] = 1.0;
    return;
  }
  E2[grp] = damp.times(s, l, [&] { return (double)s + (double)l; });
  D[grp] = (double)r + (double)c;
}

// D and lambda D^2 (a float pair) of a given float D.
__global__ void band_given_d_kernel(const float* in, BandDamping damp, double* D, float2* E2, int64_t n) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const float d = in[j], p = __fmul_rn(d, d);
  D[j] = (double)d;
  E2[j] = damp.times(p, __fmaf_rn(d, d, -p), [&] { return (double)d * (double)d; });
}

// g = J^T (b - J x) - lambda D^2 x into the parallel QR's padded layout: the residual of a row as an
// unevaluated float pair (rh + rl, Dot2: error-free products and sums, the accuracy of a double residual
// without GB300's slow FP64 pipe), the column sums as pairs too.
template <bool kW8, bool kStaged, int MW>
__global__ void __launch_bounds__(256) band_grad_f32_kernel(BandGroups B, const float* b, const float* x,
                                                            const float2* E2, bool damped,
                                                            const int64_t* blk0, float* gp) {
  dev::chain_wait();
  extern __shared__ __align__(16) float sm_f[];
  const int nt = blockDim.x, tid = threadIdx.x, w = B.w;
  const int64_t grp0 = (int64_t)blockIdx.x * (nt - (w - 1)) - (w - 1), grp = grp0 + tid;
  const float* rows = group_rows_f32<kStaged>(B.J, grp0, B.total_cols, B.rpc * w, B.gs, sm_f);
  float* xs = sm_f + (kStaged ? nt * B.gs : 0);                    // x of columns grp0 .. grp0 + nt + w - 2
  float2* S = reinterpret_cast<float2*>(xs + ((nt + w + 2) & ~3));  // per group and diagonal, stride w + 1
  for (int e = tid; e < nt + w - 1; e += nt) {
    const int64_t c = grp0 + e;
    xs[e] = c >= 0 && c < B.total_cols ? x[c] : 0.f;
  }
  const int64_t k = instance_of_group(B.inst_col0, B.inst_cols, B.num_inst, grp0, grp);   // and the staged data
  const bool have = grp >= 0 && grp < B.total_cols;
  float hs[8], hc[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) hs[t] = hc[t] = 0.f;
  if (have) {
    const int64_t left = B.inst_col0[k] + B.inst_cols[k] - grp;   // columns from the group's to the instance's end
    const int nx = left < w ? (int)left : w;
    float xv[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) xv[t] = t < nx ? -xs[tid + t] : 0.f;
    if constexpr (kW8) {
      // two entries at a time; the even and the odd entries' residual sums are added at the end of the row
      dev::f2 x2[4], nx2[4], h2[4], l2[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        x2[t] = dev::pack2(xv[2 * t], xv[2 * t + 1]);
        nx2[t] = dev::pack2(-xv[2 * t], -xv[2 * t + 1]);
        h2[t] = l2[t] = 0ull;
      }
      for (int q = 0; q < B.rpc; ++q) {
        dev::f2 a[4];
        const ulonglong2* row = reinterpret_cast<const ulonglong2*>(rows + 8 * q);
        const ulonglong2 lo = row[0], hi = row[1];
        a[0] = lo.x;
        a[1] = lo.y;
        a[2] = hi.x;
        a[3] = hi.y;
        if (nx < 8) {   // an entry past the instance's last column belongs to no column
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            float u, v;
            dev::unpack2(a[t], u, v);
            a[t] = dev::pack2(2 * t < nx ? u : 0.f, 2 * t + 1 < nx ? v : 0.f);
          }
        }
        dev::f2 sh = dev::pack2(b[grp * B.rpc + q], 0.f), sl = 0ull;
#pragma unroll
        for (int t = 0; t < 4; ++t) dev::dot2_add2(sh, sl, a[t], x2[t], nx2[t]);
        float he, ho, s, e;
        dev::unpack2(sh, he, ho);
        dev::two_sum(he, ho, s, e);
        const float c = dev::sum2(sl) + e;
        const dev::f2 s2 = dev::pack2(s, s), ns2 = dev::pack2(-s, -s), c2 = dev::pack2(c, c);
#pragma unroll
        for (int t = 0; t < 4; ++t) dev::dot2_add2(h2[t], l2[t], a[t], s2, ns2, c2);
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        dev::unpack2(h2[t], hs[2 * t], hs[2 * t + 1]);
        dev::unpack2(l2[t], hc[2 * t], hc[2 * t + 1]);
      }
    } else {
      for (int q = 0; q < B.rpc; ++q) {
        float a[8];
        row_f32<kW8, 8>(a, rows + (int64_t)q * w, w);
        float sh = b[grp * B.rpc + q], sl = 0.f;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          if (t < nx) dev::dot2(sh, sl, a[t], xv[t]);
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          if (t < nx) {   // an entry past the instance's last column belongs to no column
            const float pr = __fmul_rn(a[t], sh);
            dev::pair_add(hs[t], hc[t], pr, __fmaf_rn(a[t], sl, __fmaf_rn(a[t], sh, -pr)));
          }
        }
      }
    }
  }
#pragma unroll
  for (int t = 0; t < 8; ++t)
    if (t < w) S[tid * (w + 1) + t] = make_float2(hs[t], hc[t]);
  __syncthreads();
  if (tid < w - 1 || !have) return;
  const int64_t j = grp - B.inst_col0[k];
  float s = 0.f, c = 0.f;
  auto diagonal = [&](int t) {
    const float2 v = S[(tid - t) * (w + 1) + t];
    dev::pair_add(s, c, v.x, v.y);
  };
  if (kW8 && j >= 7) {
#pragma unroll
    for (int t = 0; t < 8; ++t) diagonal(t);
  } else {
    for (int t = 0; t < w && t <= j; ++t) diagonal(t);
  }
  if (damped) {   // - lambda D^2 x
    const float2 e2 = E2[grp];
    const float xj = -xs[tid];
    const float q = __fmul_rn(e2.x, xj);
    const float qe = __fmaf_rn(e2.y, xj, __fmaf_rn(e2.x, xj, -q));
    dev::pair_add(s, c, q, qe);
  }
  float* out = gp + 8 * blk0[k];
  out[j] = s + c;
  if (j == B.inst_cols[k] - 1)   // the padding columns of the last block
    for (int64_t e = j + 1; e < (j + 8) / 8 * 8; ++e) out[e] = 0.f;
}

// Threads, staging and shared memory for a group of rw floats: as many groups as fit about 100 KB; groups
// of more than 700 floats are read from global memory by their threads.
struct BandLaunch {
  int nt, gs;
  bool staged, w8;
  size_t smem;
  unsigned grid;
};
static BandLaunch band_launch(const BandGroups& B, size_t per_thread, size_t fixed) {
  BandLaunch L;
  const int rw = B.rpc * B.w;
  L.staged = rw <= 700;
  L.gs = (rw & 3) == 0 ? rw + 4 : (rw | 1);   // 16-byte rows, or an odd stride: no bank conflicts
  L.nt = 256;
  while (L.staged && L.nt > 32 && (size_t)L.nt * L.gs * 4 > 80 * 1024) L.nt /= 2;
  // rows by 16-byte loads: staged rows of 8 are aligned, rows in global memory if J is
  L.w8 = B.w == 8 && (L.staged || (reinterpret_cast<uintptr_t>(B.J) & 15) == 0);
  L.smem = (L.staged ? (size_t)L.nt * L.gs * 4 : 0) + L.nt * per_thread + fixed;
  const int64_t cols = L.nt - (B.w - 1);
  L.grid = (unsigned)((B.total_cols + cols - 1) / cols);
  return L;
}

// KERNEL<w = 8 by 16-byte loads, staged, widest window>, launched by LAUNCH (start_launch or chain_launch)
#define BAND_F32_LAUNCH(ctx, LAUNCH, L, KERNEL, MW, ...)                                                                   \
  do {                                                                                                         \
    auto launch_ = [&](auto k_) -> cudaError_t {                                                               \
      if ((L).smem > 48 * 1024) {                                                                              \
        const cudaError_t e_ = cudaFuncSetAttribute(k_, cudaFuncAttributeMaxDynamicSharedMemorySize,           \
                                                    (int)(L).smem);                                            \
        if (e_ != cudaSuccess) return e_;                                                                      \
      }                                                                                                        \
      return LAUNCH((ctx)->stream, (L).grid, (L).nt, (L).smem, k_, __VA_ARGS__);                               \
    };                                                                                                         \
    QRKIT_CUDA_TRY(ctx, (L).w8 ? ((L).staged ? launch_(KERNEL<true, true, 8>) : launch_(KERNEL<true, false, 8>))  \
                               : ((L).staged ? launch_(KERNEL<false, true, MW>) : launch_(KERNEL<false, false, MW>))); \
    (ctx)->launches += 1;                                                                                      \
  } while (0)

// Refinement pieces of the parallel path for double J (float J takes the Dot2 kernels
// above), one thread per row / per column: r = b - J x in double, then
// g_j = sum_i J_ij r_i - lambda D_j^2 x_j.
template <typename T>
__global__ void band_resid_kernel(const T* J, const T* b, const T* x, const int64_t* inst_cols,
                                  const int64_t* inst_col0, const int64_t* inst_row0, int64_t num_inst,
                                  int64_t total_rows, int rpc, int w, double* r) {
  const int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= total_rows) return;
  int64_t lo = 0, hi = num_inst - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) / 2;
    if (inst_row0[mid] <= gi) lo = mid; else hi = mid - 1;
  }
  const int64_t i = gi - inst_row0[lo], N = inst_cols[lo], c0 = inst_col0[lo];
  const int64_t s = i / rpc;
  const T* row = J + gi * w;
  double acc = (double)b[gi];
  for (int t = 0; t < w && s + t < N; ++t) acc -= (double)row[t] * (double)x[c0 + s + t];
  r[gi] = acc;
}

template <typename T>
__global__ void band_g_kernel(const T* J, const T* x, const double* r, const double* D, double lam,
                              const int64_t* inst_cols, const int64_t* inst_col0, const int64_t* inst_row0,
                              int64_t num_inst, int64_t total_cols, int rpc, int w, double* g) {
  const int64_t gj = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gj >= total_cols) return;
  int64_t lo = 0, hi = num_inst - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) / 2;
    if (inst_col0[mid] <= gj) lo = mid; else hi = mid - 1;
  }
  const int64_t j = gj - inst_col0[lo], N = inst_cols[lo], r0 = inst_row0[lo];
  const int64_t nrows = (int64_t)rpc * N;
  double acc = 0.0;
  const int64_t s_lo = j - w + 1 > 0 ? j - w + 1 : 0;
  for (int64_t s = s_lo; s <= j; ++s)
    for (int q = 0; q < rpc; ++q) {
      const int64_t i = s * rpc + q;
      if (i >= nrows) break;
      acc += (double)J[(r0 + i) * w + (j - s)] * r[r0 + i];
    }
  if (lam > 0.0) acc -= lam * D[gj] * D[gj] * (double)x[gj];
  g[gj] = acc;
}

// Rows with explicit starts (global columns, non-decreasing within an instance): the rows of
// instance k are row0[k] .. row0[k] + rows[k] - 1, and column j is touched by the rows whose
// start lies in [j - w + 1, j], a contiguous run found by binary search.  inst: 4 x num_inst
// (cols, col0, row0, rows).
__device__ __forceinline__ int64_t inst_of_col(const int64_t* inst, int64_t num_inst, int64_t gj) {
  const int64_t* col0 = inst + num_inst;
  int64_t lo = 0, hi = num_inst - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) / 2;
    if (col0[mid] <= gj) lo = mid; else hi = mid - 1;
  }
  return lo;
}
// First row of [r0, r1) whose start is >= v (starts sorted in that range).
__device__ __forceinline__ int64_t first_row_at(const int64_t* start, int64_t r0, int64_t r1, int64_t v) {
  while (r0 < r1) {
    const int64_t mid = r0 + (r1 - r0) / 2;
    if (start[mid] < v) r0 = mid + 1; else r1 = mid;
  }
  return r0;
}

// D_j = || column j of J || (zero -> 1), one thread per global column, rows in order.
template <typename T>
__global__ void band_colnorm_explicit_kernel(const T* J, const int64_t* start, const int64_t* inst,
                                             int64_t num_inst, int64_t total_cols, int w, double* D) {
  const int64_t gj = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gj >= total_cols) return;
  const int64_t k = inst_of_col(inst, num_inst, gj);
  const int64_t r0 = inst[2 * num_inst + k], r1 = r0 + inst[3 * num_inst + k];
  double acc = 0.0;
  for (int64_t i = first_row_at(start, r0, r1, gj - w + 1); i < r1 && start[i] <= gj; ++i) {
    const double v = (double)J[i * w + (gj - start[i])];
    acc += v * v;
  }
  const double d = sqrt(acc);
  D[gj] = d == 0.0 ? 1.0 : d;
}

// r_i = b_i - sum_t J_it x_{start_i + t} in double (entries past the instance's last column are
// ignored), one thread per row.
template <typename T>
__global__ void band_resid_explicit_kernel(const T* J, const T* b, const T* x, const int64_t* start,
                                           const int64_t* inst, int64_t num_inst, int64_t total_rows, int w,
                                           double* r) {
  const int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= total_rows) return;
  const int64_t* row0 = inst + 2 * num_inst;
  int64_t lo = 0, hi = num_inst - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) / 2;
    if (row0[mid] <= gi) lo = mid; else hi = mid - 1;
  }
  const int64_t end = inst[num_inst + lo] + inst[lo];   // one past the instance's last column
  double acc = (double)b[gi];
  for (int t = 0; t < w && start[gi] + t < end; ++t) acc -= (double)J[gi * w + t] * (double)x[start[gi] + t];
  r[gi] = acc;
}

// g_j = sum_i J_ij r_i - lambda D_j^2 x_j, one thread per global column, rows in order.
template <typename T>
__global__ void band_g_explicit_kernel(const T* J, const T* x, const double* r, const double* D, double lam,
                                       const int64_t* start, const int64_t* inst, int64_t num_inst,
                                       int64_t total_cols, int w, double* g) {
  const int64_t gj = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gj >= total_cols) return;
  const int64_t k = inst_of_col(inst, num_inst, gj);
  const int64_t r0 = inst[2 * num_inst + k], r1 = r0 + inst[3 * num_inst + k];
  double acc = 0.0;
  for (int64_t i = first_row_at(start, r0, r1, gj - w + 1); i < r1 && start[i] <= gj; ++i)
    acc += (double)J[i * w + (gj - start[i])] * r[i];
  if (lam > 0.0) acc -= lam * D[gj] * D[gj] * (double)x[gj];
  g[gj] = acc;
}

template <typename T>
__global__ void band_axpy_kernel(T* x, const T* d, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] += d[i];
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

qrkit_status banded_plan(qrkit_ctx* ctx, const qrkit_structure* s) {
  Plan& P = ctx->plan;
  if (s->rows_per_col < 1) return fail(ctx, QRKIT_EINVAL, "rows_per_col must be >= 1");
  if (s->band_window < 1 || s->band_window > kBW)
    return fail(ctx, QRKIT_EUNSUPPORTED, "band_window must be in [1, 16]");
  std::vector<int64_t> cols;
  if (s->num_blocks > 0 && s->instance_cols) {
    cols.assign(s->instance_cols, s->instance_cols + s->num_blocks);
  } else {
    if (s->cols < 1) return fail(ctx, QRKIT_EINVAL, "cols must be >= 1");
    cols.assign(1, s->cols);
  }
  for (size_t i = 0; i < cols.size(); ++i)
    if (cols[i] < 1) return fail(ctx, QRKIT_EINVAL, "instance " + std::to_string(i) + " has no columns");
  // rows per instance: rows_per_col * cols, or given with explicit row starts
  const bool expl = s->band_row_start != nullptr;
  std::vector<int64_t> nrows(cols.size());
  for (size_t i = 0; i < cols.size(); ++i) {
    if (!expl) {
      nrows[i] = cols[i] * s->rows_per_col;
    } else if (s->instance_rows) {
      nrows[i] = s->instance_rows[i];
    } else if (cols.size() == 1) {
      nrows[i] = s->rows;
    } else {
      return fail(ctx, QRKIT_EINVAL, "instance_rows is required with band_row_start and a batch of instances");
    }
    if (nrows[i] < 0) return fail(ctx, QRKIT_EINVAL, "instance " + std::to_string(i) + " has a negative row count");
  }
  std::vector<int64_t> c0(cols.size()), r0(cols.size());
  int64_t cc = 0, rr = 0;
  for (size_t i = 0; i < cols.size(); ++i) {
    c0[i] = cc;
    r0[i] = rr;
    cc += cols[i];
    rr += nrows[i];
  }
  std::vector<int64_t> gstart;
  if (expl) {
    gstart.resize((size_t)rr);
    for (size_t i = 0; i < cols.size(); ++i)
      for (int64_t k = 0; k < nrows[i]; ++k) {
        const int64_t v = s->band_row_start[r0[i] + k];
        if (v < 0 || v >= cols[i])
          return fail(ctx, QRKIT_EINVAL, "row " + std::to_string(r0[i] + k) + " starts outside its instance");
        if (k > 0 && v < s->band_row_start[r0[i] + k - 1])
          return fail(ctx, QRKIT_EINVAL, "row starts must not decrease within an instance (row " +
                                             std::to_string(r0[i] + k) + ")");
        gstart[(size_t)(r0[i] + k)] = c0[i] + v;
      }
  }
  Band& B = ctx->band;
  if (s->band_solver < QRKIT_BAND_AUTO || s->band_solver > QRKIT_BAND_PARALLEL)
    return fail(ctx, QRKIT_EINVAL, "unknown band_solver");
  if (s->band_solver == QRKIT_BAND_PARALLEL && s->band_window > 8)
    return fail(ctx, QRKIT_EUNSUPPORTED, "the parallel banded QR needs band_window <= 8");
  B.parallel = s->band_solver == QRKIT_BAND_PARALLEL || (s->band_solver == QRKIT_BAND_AUTO && s->band_window <= 8);
  B.num_inst = (int64_t)cols.size();
  B.total_cols = cc;
  B.total_rows = rr;
  B.rows_per_col = s->rows_per_col;
  B.w = s->band_window;
  B.explicit_starts = expl;
  qrkit_status st;
  auto up = [&](DevBuf& buf, const std::vector<int64_t>& v) -> qrkit_status {
    qrkit_status r = ensure(ctx, buf, v.size() * sizeof(int64_t), "band plan");
    if (r != QRKIT_OK) return r;
    QRKIT_CUDA_TRY(ctx, cudaMemcpy(buf.ptr, v.data(), v.size() * sizeof(int64_t), cudaMemcpyHostToDevice));
    return QRKIT_OK;
  };
  if ((st = up(B.d_cols, cols)) != QRKIT_OK) return st;
  if ((st = up(B.d_col0, c0)) != QRKIT_OK) return st;
  if ((st = up(B.d_row0, r0)) != QRKIT_OK) return st;
  if (expl) {
    std::vector<int64_t> inst(cols);
    inst.insert(inst.end(), c0.begin(), c0.end());
    inst.insert(inst.end(), r0.begin(), r0.end());
    inst.insert(inst.end(), nrows.begin(), nrows.end());
    if ((st = up(B.d_inst, inst)) != QRKIT_OK) return st;
    if ((st = up(B.d_rows, nrows)) != QRKIT_OK) return st;
    if (rr > 0 && (st = up(B.d_start, gstart)) != QRKIT_OK) return st;
  }
  const size_t es = elem_size(ctx);
  if ((st = ensure(ctx, B.Rw, (size_t)cc * B.w * es, "banded R")) != QRKIT_OK) return st;
  if ((st = ensure(ctx, B.c, (size_t)cc * es, "banded c")) != QRKIT_OK) return st;
  if ((st = ensure(ctx, B.D, (size_t)cc * sizeof(double), "banded D")) != QRKIT_OK) return st;
  if (es == sizeof(float) && (st = ensure(ctx, B.E2, (size_t)cc * sizeof(float2), "banded D")) != QRKIT_OK) return st;
  if ((st = ensure(ctx, B.res2, (size_t)B.num_inst * sizeof(double), "banded residual")) != QRKIT_OK) return st;
  if (B.parallel) {
    if ((st = cr_build(ctx, B.cr, cols, c0, r0, nrows)) != QRKIT_OK) return st;
  }
  if (expl || (B.parallel && ctx->precision == QRKIT_FP64)) {   // the float gradient needs no scratch
    if ((st = ensure(ctx, B.g, (size_t)cc * sizeof(double), "banded g")) != QRKIT_OK) return st;
    if ((st = ensure(ctx, B.h, (size_t)cc * es, "banded h")) != QRKIT_OK) return st;
    if ((st = ensure(ctx, B.r, (size_t)std::max<int64_t>(rr, 1) * sizeof(double), "banded r")) != QRKIT_OK) return st;
  }
  P.s = *s;
  P.s.block_rows = nullptr;
  P.s.block_cols = nullptr;
  P.s.window_start = nullptr;
  P.s.instance_cols = nullptr;
  P.s.band_row_start = nullptr;
  P.s.instance_rows = nullptr;
  P.valid = true;
  return QRKIT_OK;
}

template <typename T>
__global__ void band_g_to_t_kernel(const double* g, T* h, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) h[i] = (T)g[i];
}

static qrkit_status widen_or_narrow_g(qrkit_ctx* ctx, const double* g, void* h, int64_t n) {
  if (ctx->precision == QRKIT_FP64)
    band_g_to_t_kernel<double><<<nblk(n, 256), 256, 0, ctx->stream>>>(g, (double*)h, n);
  else
    band_g_to_t_kernel<float><<<nblk(n, 256), 256, 0, ctx->stream>>>(g, (float*)h, n);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}

template <typename T>
static qrkit_status banded_run(qrkit_ctx* ctx, const void* J, const void* b, const void* Dext,
                               double lambda, void* p, int refine_steps) {
  Band& B = ctx->band;
  cudaStream_t st = ctx->stream;
  const int64_t* dcols = (const int64_t*)B.d_cols.ptr;
  const int64_t* dc0 = (const int64_t*)B.d_col0.ptr;
  const int64_t* dr0 = (const int64_t*)B.d_row0.ptr;
  double* D = (double*)B.D.ptr;
  if (lambda > 0.0) {
    if (Dext) {
      if (sizeof(T) == sizeof(double)) {
        QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(D, Dext, (size_t)B.total_cols * sizeof(double),
                                            cudaMemcpyDeviceToDevice, st));
      } else {
        band_given_d_kernel<<<nblk(B.total_cols, 256), 256, 0, st>>>((const float*)Dext, BandDamping(lambda), D,
                                                                    (float2*)B.E2.ptr, B.total_cols);
        ctx->launches += 1;
        QRKIT_CUDA_TRY(ctx, cudaGetLastError());
      }
    } else if (B.explicit_starts) {
      band_colnorm_explicit_kernel<T><<<nblk(B.total_cols, 256), 256, 0, st>>>(
          (const T*)J, (const int64_t*)B.d_start.ptr, (const int64_t*)B.d_inst.ptr, B.num_inst, B.total_cols, B.w,
          D);
      ctx->launches += 1;
      QRKIT_CUDA_TRY(ctx, cudaGetLastError());
    } else {
      if (sizeof(T) == sizeof(float)) {
        const BandGroups G{(const float*)J, B.total_cols, dcols, dc0, B.num_inst, B.rows_per_col, B.w, 0};
        const BandLaunch L = band_launch(G, (size_t)(B.w + 1) * sizeof(float), 0);
        BandGroups GL = G;
        GL.gs = L.gs;
        const BandDamping damp(lambda);
        if (B.w <= 8) BAND_F32_LAUNCH(ctx, start_launch, L, band_norm_f32_kernel, 8, GL, damp, D, (float2*)B.E2.ptr);
        else BAND_F32_LAUNCH(ctx, start_launch, L, band_norm_f32_kernel, kBW, GL, damp, D, (float2*)B.E2.ptr);
      } else {
        band_colnorm_kernel<<<nblk(B.total_cols, 256), 256, 0, st>>>(nullptr, (const double*)J, dcols, dc0, dr0,
                                                                    B.num_inst, B.rows_per_col, B.w, D);
        ctx->launches += 1;
        QRKIT_CUDA_TRY(ctx, cudaGetLastError());
      }
    }
  }
  if (B.explicit_starts) {
    // rows with explicit starts (e.g. the row and column permutations of Sec. 4.3 applied):
    // the parallel QR or the sweep, then refinement with a double residual
    const int64_t* gs = (const int64_t*)B.d_start.ptr;
    const int64_t* inst = (const int64_t*)B.d_inst.ptr;
    qrkit_status rc;
    if (B.parallel) {
      rc = cr_solve(ctx, *B.cr, gs, nullptr, 1, B.w, J, b, D, lambda, p, (double*)B.res2.ptr);
    } else {
      rc = banded_explicit_solve(ctx, B.num_inst, inst, J, gs, b, B.w, D, lambda, B.Rw.ptr, B.c.ptr, p,
                                 (double*)B.res2.ptr);
    }
    if (rc != QRKIT_OK) return rc;
    for (int it = 0; it < refine_steps; ++it) {
      band_resid_explicit_kernel<T><<<nblk(std::max<int64_t>(B.total_rows, 1), 256), 256, 0, st>>>(
          (const T*)J, (const T*)b, (const T*)p, gs, inst, B.num_inst, B.total_rows, B.w, (double*)B.r.ptr);
      band_g_explicit_kernel<T><<<nblk(B.total_cols, 256), 256, 0, st>>>(
          (const T*)J, (const T*)p, (const double*)B.r.ptr, D, lambda, gs, inst, B.num_inst, B.total_cols, B.w,
          (double*)B.g.ptr);
      ctx->launches += 2;
      QRKIT_CUDA_TRY(ctx, cudaGetLastError());
      if (B.parallel) {
        if ((rc = cr_normal_solve(ctx, *B.cr, (const double*)B.g.ptr, nullptr, p)) != QRKIT_OK) return rc;
        continue;
      } else {
        if ((rc = widen_or_narrow_g(ctx, (const double*)B.g.ptr, B.h.ptr, B.total_cols)) != QRKIT_OK) return rc;
        if ((rc = banded_tri_solve(ctx, B.num_inst, inst, B.Rw.ptr, B.w, B.h.ptr, true)) != QRKIT_OK) return rc;
        if ((rc = banded_tri_solve(ctx, B.num_inst, inst, B.Rw.ptr, B.w, B.h.ptr, false)) != QRKIT_OK) return rc;
      }
      band_axpy_kernel<T><<<nblk(B.total_cols, 256), 256, 0, st>>>((T*)p, (const T*)B.h.ptr, B.total_cols);
      ctx->launches += 1;
      QRKIT_CUDA_TRY(ctx, cudaGetLastError());
    }
    return QRKIT_OK;
  }
  if (B.parallel) {
    qrkit_status rc = cr_solve(ctx, *B.cr, nullptr, nullptr, B.rows_per_col, B.w, J, b, D, lambda, p,
                               (double*)B.res2.ptr);
    if (rc != QRKIT_OK) return rc;
    for (int it = 0; it < refine_steps; ++it) {
      if constexpr (sizeof(T) == sizeof(float)) {
        const BandGroups G{(const float*)J, B.total_cols, dcols, dc0, B.num_inst, B.rows_per_col, B.w, 0};
        const BandLaunch L = band_launch(G, (size_t)(B.w + 1) * sizeof(float2) + sizeof(float), (B.w + 3) * sizeof(float));
        BandGroups GL = G;
        GL.gs = L.gs;
        const int64_t* blk0;
        void* gp;
        cr_padded(*B.cr, &blk0, &gp);
        BAND_F32_LAUNCH(ctx, chain_launch, L, band_grad_f32_kernel, 8, GL, (const float*)b, (const float*)p,
                        (const float2*)B.E2.ptr, lambda > 0.0, blk0, (float*)gp);
      } else {
        band_resid_kernel<T><<<nblk(B.total_rows, 256), 256, 0, st>>>(
            (const T*)J, (const T*)b, (const T*)p, dcols, dc0, dr0, B.num_inst, B.total_rows, B.rows_per_col, B.w,
            (double*)B.r.ptr);
        band_g_kernel<T><<<nblk(B.total_cols, 256), 256, 0, st>>>(
            (const T*)J, (const T*)p, (const double*)B.r.ptr, D, lambda, dcols, dc0, dr0, B.num_inst, B.total_cols,
            B.rows_per_col, B.w, (double*)B.g.ptr);
        ctx->launches += 2;
        QRKIT_CUDA_TRY(ctx, cudaGetLastError());
      }
      if ((rc = cr_normal_solve(ctx, *B.cr, sizeof(T) == sizeof(float) ? nullptr : (const double*)B.g.ptr, nullptr, p)) !=
          QRKIT_OK)
        return rc;
    }
    return QRKIT_OK;
  }
  BandArgs<T> A;
  A.num_inst = B.num_inst;
  A.inst_cols = dcols;
  A.inst_col0 = dc0;
  A.inst_row0 = dr0;
  A.rows_per_col = B.rows_per_col;
  A.row_start = nullptr;
  A.inst_rows = nullptr;
  A.w = B.w;
  A.J = (const T*)J;
  A.b = (const T*)b;
  A.D = D;
  A.lam = lambda;
  A.Rw = (T*)B.Rw.ptr;
  A.c = (T*)B.c.ptr;
  A.x = (T*)p;
  A.res2 = (double*)B.res2.ptr;
  A.refine_steps = refine_steps;
  A.status = ctx->d_status;
  banded_factor_solve_kernel<T><<<nblk(B.num_inst, warps_for<T>()), 32 * warps_for<T>(), 0, st>>>(A);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  if constexpr (sizeof(T) == sizeof(float)) {
    if (refine_steps > 0) {
      qrkit_status rc;
      if ((rc = ensure(ctx, B.g, (size_t)B.total_cols * sizeof(double), "banded g")) != QRKIT_OK) return rc;
      if ((rc = ensure(ctx, B.h, (size_t)B.total_cols * sizeof(float), "banded h")) != QRKIT_OK) return rc;
      if ((rc = ensure(ctx, B.r, (size_t)B.total_rows * sizeof(double), "banded r")) != QRKIT_OK) return rc;
      for (int it = 0; it < refine_steps; ++it) {
        banded_refine_kernel<<<nblk(B.num_inst, kWarps), 32 * kWarps, 0, st>>>(
            A, (double*)B.r.ptr, (double*)B.g.ptr, (float*)B.h.ptr);
        ctx->launches += 1;
        QRKIT_CUDA_TRY(ctx, cudaGetLastError());
      }
    }
  }
  return QRKIT_OK;
}

// Factor + solve banded instances whose rows carry explicit starts (the reduced blocks of a
// windowed block-angular structure, one instance per segment of S): rows x w values, damping
// rows lambda^(1/2) D_j (D in double, global columns) when lambda > 0.  Rw, c, x, D are
// indexed by global column (instance col0 + j); rows, starts and rhs by global row.
template <typename T>
static qrkit_status explicit_run(qrkit_ctx* ctx, int64_t num_inst, const int64_t* inst, const T* rows,
                                 const int64_t* starts, const T* rhs, int w, const double* D,
                                 double lambda, T* Rw, T* c, T* x, double* res2) {
  BandArgs<T> A;
  A.num_inst = num_inst;
  A.inst_cols = inst;
  A.inst_col0 = inst + num_inst;
  A.inst_row0 = inst + 2 * num_inst;
  A.inst_rows = inst + 3 * num_inst;
  A.rows_per_col = 1;
  A.row_start = starts;
  A.w = w;
  A.J = rows;
  A.b = rhs;
  A.D = D;
  A.lam = lambda;
  A.Rw = Rw;
  A.c = c;
  A.x = x;
  A.res2 = res2;
  A.refine_steps = 0;
  A.status = ctx->d_status;
  banded_factor_solve_kernel<T><<<nblk(num_inst, warps_for<T>()), 32 * warps_for<T>(), 0, ctx->stream>>>(A);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}

qrkit_status banded_explicit_solve(qrkit_ctx* ctx, int64_t num_inst, const int64_t* inst,
                                   const void* rows, const int64_t* starts, const void* rhs, int w,
                                   const double* D, double lambda, void* Rw, void* c, void* x,
                                   double* res2) {
  if (w < 1 || w > kBW) return fail(ctx, QRKIT_EUNSUPPORTED, "reduced band window must be in [1, 16]");
  if (num_inst < 1) return QRKIT_OK;
  if (ctx->precision == QRKIT_FP64)
    return explicit_run<double>(ctx, num_inst, inst, (const double*)rows, starts, (const double*)rhs, w,
                                D, lambda, (double*)Rw, (double*)c, (double*)x, res2);
  return explicit_run<float>(ctx, num_inst, inst, (const float*)rows, starts, (const float*)rhs, w, D,
                             lambda, (float*)Rw, (float*)c, (float*)x, res2);
}

qrkit_status banded_tri_solve(qrkit_ctx* ctx, int64_t num_inst, const int64_t* inst, const void* Rw,
                              int w, void* v, bool transpose) {
  if (num_inst < 1) return QRKIT_OK;
  if (ctx->precision == QRKIT_FP64)
    band_tri_solve_kernel<double><<<nblk(num_inst, 64), 64, 0, ctx->stream>>>(
        num_inst, inst, (const double*)Rw, w, (double*)v, transpose ? 1 : 0);
  else
    band_tri_solve_kernel<float><<<nblk(num_inst, 64), 64, 0, ctx->stream>>>(
        num_inst, inst, (const float*)Rw, w, (float*)v, transpose ? 1 : 0);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}

qrkit_status banded_factor_solve(qrkit_ctx* ctx, const void* J, const void* b, const void* D,
                                 double lambda, void* p, int refine_steps) {
  if (ctx->precision == QRKIT_FP64) return banded_run<double>(ctx, J, b, D, lambda, p, 0);
  const int steps = ctx->precision == QRKIT_FP32 ? 0 : refine_steps;
  return banded_run<float>(ctx, J, b, D, lambda, p, steps);
}

qrkit_status banded_get_factor(qrkit_ctx* ctx, void* Rw_out, void* c_out, double* res2_out) {
  Band& B = ctx->band;
  const size_t es = elem_size(ctx);
  if (B.parallel && (Rw_out || c_out))
    return fail(ctx, QRKIT_EUNSUPPORTED, "R windows and Q^T b exist only for the sweep algorithm");
  if (Rw_out)
    QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(Rw_out, B.Rw.ptr, (size_t)B.total_cols * B.w * es,
                                        cudaMemcpyDeviceToDevice, ctx->stream));
  if (c_out)
    QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(c_out, B.c.ptr, (size_t)B.total_cols * es,
                                        cudaMemcpyDeviceToDevice, ctx->stream));
  if (res2_out)
    QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(res2_out, B.res2.ptr, (size_t)B.num_inst * sizeof(double),
                                        cudaMemcpyDeviceToHost, ctx->stream));
  return QRKIT_OK;
}

void release_band(Band& B) {
  release(B.d_cols); release(B.d_col0); release(B.d_row0); release(B.Rw); release(B.c);
  release(B.d_inst); release(B.d_rows); release(B.d_start);
  release(B.D); release(B.E2); release(B.res2); release(B.g); release(B.h); release(B.r);
  release_cr(B.cr);
  B = Band();
}

}  // namespace qrkit
