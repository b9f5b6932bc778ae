// Solves with a dense shared part S (Sec. 4.2, Sec. 5.1): the triangle R_S of the reduced block,
// the block unknowns below it, and the refinement residual of float plans.
//
// Every pass over S (column-major, rows of J) or R12 (row-major, one row of s values per block
// column) is written for the memory system: a warp reads whole 128-byte lines, a CTA's warps split
// the columns, sums leave through per-chunk partials that are added in a fixed order.  S and R12
// are read twice and once per refinement step; those passes are bound by HBM and by the additions of the
// three-float sums (22 and 33 operations per value): at 100,000 blocks
// 4 x 2 with s = 512 (S 819 MB, R12 410 MB) the row pass takes 186 us, the column pass 250 us, the
// R12 pass 159 us (126, 135 and 136 with float pairs, which are not enough: see the refinement below) and a block
// back-substitution 95 us.  A thread per block walking all s columns,
// with a shared-memory FP64 atomic per column and block, took 4.33 ms for the two passes over S,
// 4.04 ms for R12^T h and 0.38 ms per back-substitution.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "chain.cuh"
#include "device_util.cuh"
#include "internal.h"
#include "sums.cuh"

namespace qrkit {
namespace {

// A double as a sum of three floats, and back.
__device__ __forceinline__ dev::Triple triple_of(double v) {
  dev::Triple s;
  s.h = (float)v;
  s.l = (float)(v - (double)s.h);
  s.m = (float)(v - (double)s.h - (double)s.l);
  return s;
}

template <int V>
struct Vec;
template <>
struct Vec<4> {
  float v[4];
  __device__ __forceinline__ void load(const float* p) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  }
};
template <>
struct Vec<1> {
  float v[1];
  __device__ __forceinline__ void load(const float* p) { v[0] = *p; }
};

// ---- triangular solves with R_S: one CTA, thread i owns row (or column) i, 32 at a time ----
// The 32 unknowns of a diagonal block are found by the warp that owns them (broadcasts, no
// barrier); then every other thread takes their 32 products off its own right-hand side in one
// go, its 32 values of R fetched while the diagonal block is being solved.  Two barriers per 32
// columns instead of one or two per column (s = 512: 82 us against 211 us for R_S x = c, 240 us
// against 465 us for R_S^T and R_S together).
constexpr int kTriThreads = kMaxDenseS;
inline unsigned tri_cta(int s) { return (unsigned)((s + 31) / 32 * 32); }

// R x = y (upper triangular, column-major): returns x_i for thread i < s; xs: 32 shared values.
template <typename T>
__device__ __forceinline__ T tri_backsub(const T* R, int64_t ld, int s, T y, T* xs, int* status) {
  const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
  T r[32];
  for (int kb = (s - 1) / 32; kb >= 0; --kb) {
    const int k0 = kb * 32, nk = min(32, s - k0);
    if (warp <= kb) {
#pragma unroll
      for (int j = 0; j < 32; ++j) r[j] = (j < nk && i <= k0 + j) ? R[(int64_t)(k0 + j) * ld + i] : T(0);
    }
    if (warp == kb) {
      T x = T(0);
#pragma unroll
      for (int j = 31; j >= 0; --j) {
        if (j < nk) {
          if (lane == j) {
            if (r[j] == T(0)) dev::record(status, QRKIT_ESINGULAR);
            x = y / r[j];
          }
          const T xj = __shfl_sync(0xffffffffu, x, j);
          if (lane < j) y -= r[j] * xj;
        }
      }
      y = x;
      xs[lane] = x;
    }
    __syncthreads();
    if (warp < kb) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (j < nk) y -= r[j] * xs[j];
    }
    __syncthreads();
  }
  return y;
}

// R^T h = g: returns h_i for thread i < s.
template <typename T>
__device__ __forceinline__ T tri_fwdsub(const T* R, int64_t ld, int s, T g, T* xs) {
  const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
  T r[32];
  for (int kb = 0; kb * 32 < s; ++kb) {
    const int k0 = kb * 32, nk = min(32, s - k0);
    if (warp >= kb) {
#pragma unroll
      for (int j = 0; j < 32; ++j) r[j] = (j < nk && i < s && k0 + j <= i) ? R[(int64_t)i * ld + k0 + j] : T(0);
    }
    if (warp == kb) {
      T x = T(0);
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        if (j < nk) {
          if (lane == j) x = g / r[j];
          const T xj = __shfl_sync(0xffffffffu, x, j);
          if (lane > j) g -= r[j] * xj;
        }
      }
      g = x;
      xs[lane] = x;
    }
    __syncthreads();
    if (warp > kb) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (j < nk) g -= r[j] * xs[j];
    }
    __syncthreads();
  }
  return g;
}

// x = R_S^{-1} c (x may be c).
template <typename T>
__global__ void __launch_bounds__(kTriThreads) tri_backsub_kernel(const T* R, int64_t ld, int s, const T* c, T* x,
                                                                  int* status) {
  dev::chain_wait();
  __shared__ T xs[32];
  const int i = threadIdx.x;
  const T y = tri_backsub<T>(R, ld, s, i < s ? c[i] : T(0), xs, status);
  if (i < s) x[i] = y;
}

// dp = R_S^{-1} R_S^{-T} g (g in double), written to dp and added to x.
template <typename T>
__global__ void __launch_bounds__(kTriThreads) tri_normal_kernel(const T* R, int64_t ld, int s, const double* g, T* dp,
                                                                 T* x, int* status) {
  dev::chain_wait();
  __shared__ T xs[32];
  const int i = threadIdx.x;
  const T h = tri_fwdsub<T>(R, ld, s, i < s ? (T)g[i] : T(0), xs);
  const T y = tri_backsub<T>(R, ld, s, h, xs, status);
  if (i < s) {
    dp[i] = y;
    x[i] += y;
  }
}

// y := R^-1 y with R = F's leading m x m upper triangle (m <= 8, columns of na).
template <typename T>
__device__ __forceinline__ void block_substitute(const T* F, int na, int m, T (&y)[8]) {
#pragma unroll
  for (int k = 7; k >= 0; --k) {
    if (k < m) {
      T v = y[k];
#pragma unroll
      for (int j = k + 1; j < 8; ++j)
        if (j < m) v -= F[j * na + k] * y[j];
      y[k] = v / F[k * na + k];
    }
  }
}

// ---- block unknowns R_i x_i = c_i - R12_i x_S, one warp per block ----
// The lanes share a row of R12 (s values, contiguous), so that the pass over R12 is coalesced and
// many loads are in flight; the m_i <= 8 unknowns are then found by every lane alike.
constexpr int kWarpBackThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kWarpBackThreads) block_backsub_warp_kernel(ComposedView<T> V, FactorOut<T> O,
                                                                              const T* rhs, const T* xS, T* x,
                                                                              int accumulate) {
  dev::chain_wait();
  __shared__ __align__(16) T xs[kMaxDenseS];
  const int s = V.s;
  for (int t = threadIdx.x; t < s; t += kWarpBackThreads) xs[t] = xS[t];
  __syncthreads();
  const int64_t i = ((int64_t)blockIdx.x * kWarpBackThreads + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= V.K) return;
  const int n = V.n[i], m = V.m[i];
  const int na = n + (O.damp ? m : 0);
  const int64_t c0 = V.col_off[i];
  const T* F = O.Fa + O.aug_off[i];
  T y[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    y[k] = T(0);
    if (k < m) {
      const T* r12 = O.R12 + (c0 + k) * (int64_t)s;
      T a = T(0);
      bool done = false;
      if constexpr (sizeof(T) == 4) {
        if ((s & 3) == 0) {   // rows of R12 are then 16-byte aligned
          const float4* r4 = reinterpret_cast<const float4*>(r12);
          const float4* x4 = reinterpret_cast<const float4*>(xs);
#pragma unroll 4
          for (int t = lane; t < s / 4; t += 32) {
            const float4 q = r4[t], z = x4[t];
            a += q.x * z.x + q.y * z.y + q.z * z.z + q.w * z.w;
          }
          done = true;
        }
      }
      if (!done)
        for (int t = lane; t < s; t += 32) a += r12[t] * xs[t];
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
      y[k] = rhs[c0 + k] - a;
    }
  }
  __syncwarp();   // x may be rhs: every lane has read it
  block_substitute(F, na, m, y);
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (k < m && lane == k) x[c0 + k] = accumulate ? x[c0 + k] + y[k] : y[k];
}

// The same with a thread per block, for many blocks.  Eight partial sums keep as many loads in flight and the sum of s
// products as accurate as the warp's.
constexpr int kThreadBackThreads = 64;

template <typename T>
__global__ void __launch_bounds__(kThreadBackThreads) block_backsub_thread_kernel(ComposedView<T> V, FactorOut<T> O,
                                                                                  const T* rhs, const T* xS, T* x,
                                                                                  int accumulate) {
  dev::chain_wait();
  __shared__ T xs[kMaxDenseS];
  const int s = V.s;
  for (int t = threadIdx.x; t < s; t += kThreadBackThreads) xs[t] = xS[t];
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * kThreadBackThreads + threadIdx.x;
  if (i >= V.K) return;
  const int n = V.n[i], m = V.m[i];
  const int na = n + (O.damp ? m : 0);
  const int64_t c0 = V.col_off[i];
  T y[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    y[k] = T(0);
    if (k < m) {
      const T* r12 = O.R12 + (c0 + k) * (int64_t)s;
      T a[8] = {};
      for (int t = 0; t < s; t += 8)
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (t + j < s) a[j] += r12[t + j] * xs[t + j];
      y[k] = rhs[c0 + k] - (((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7])));
    }
  }
  block_substitute(O.Fa + O.aug_off[i], na, m, y);
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (k < m) x[c0 + k] = accumulate ? x[c0 + k] + y[k] : y[k];
}

// ---- refinement of float plans: g = J^T (b - J p - S p_S) - lambda D^2 p with the residual and its sums as sums of
// three floats, no less accurate than in double: with a residual 1e9 times what the unknowns explain, float pairs left
// the refined solution off by 1.3e-7 to 2.1e-7, sums in double and these by 2.5e-8.  A product that overflows (right-hand sides have any scale) leaves a
// sum that is not finite: that one is formed again in double. ----

// 1. rows: b - S p_S, three floats per row.  A CTA takes 32 V rows; its 8 warps split the columns.
constexpr int kRowWarps = 8;

template <int V>
__global__ void __launch_bounds__(32 * kRowWarps) dense_rows_kernel(const float* S, int64_t rows, int s, const float* b,
                                                                    const float* pS, float* rh, float* rl, float* rm) {
  dev::chain_wait();
  __shared__ float part[3][kRowWarps][32 * V];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t row0 = (int64_t)blockIdx.x * (32 * V);
  const int64_t row = row0 + lane * V;
  dev::Triple sum[V];
  if (row < rows) {   // V divides rows
    const float* src = S + row;
    int c = warp;
    for (; c + 3 * kRowWarps < s; c += 4 * kRowWarps) {
      Vec<V> a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u].load(src + (int64_t)(c + u * kRowWarps) * rows);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float p = -pS[c + u * kRowWarps];
#pragma unroll
        for (int q = 0; q < V; ++q) sum[q].fma(a[u].v[q], p);
      }
    }
    for (; c < s; c += kRowWarps) {
      Vec<V> a;
      a.load(src + (int64_t)c * rows);
      const float p = -pS[c];
#pragma unroll
      for (int q = 0; q < V; ++q) sum[q].fma(a.v[q], p);
    }
  }
#pragma unroll
  for (int q = 0; q < V; ++q) {
    part[0][warp][lane * V + q] = sum[q].h;
    part[1][warp][lane * V + q] = sum[q].l;
    part[2][warp][lane * V + q] = sum[q].m;
  }
  __syncthreads();
  const int t = threadIdx.x;
  if (t < 32 * V && row0 + t < rows) {
    dev::Triple r;
    r.h = b[row0 + t];
#pragma unroll
    for (int w = 0; w < kRowWarps; ++w) r.add(part[0][w][t], part[1][w][t], part[2][w][t]);
    if (!isfinite(r.h + r.l)) {
      double v = (double)b[row0 + t];
      for (int c = 0; c < s; ++c) v -= (double)S[(int64_t)c * rows + row0 + t] * (double)pS[c];
      r = triple_of(v);
    }
    rh[row0 + t] = r.h;
    rl[row0 + t] = r.l;
    rm[row0 + t] = r.m;
  }
}

// 2. blocks (one thread each): r -= J p, g_B = J^T r - lambda D^2 p, h_B = R_i^{-T} g_B.
__global__ void __launch_bounds__(128) dense_blocks_kernel(ComposedView<float> V, FactorOut<float> O, const float* p,
                                                           double lam, float* rh, float* rl, float* rm, float* h) {
  dev::chain_wait();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= V.K) return;
  const int n = V.n[i], m = V.m[i];
  const int na = n + (O.damp ? m : 0);
  const int64_t c0 = V.col_off[i], r0 = V.row_off[i];
  const float* J = V.J + V.val_off[i];
  const float* F = O.Fa + O.aug_off[i];
  float pj[8], hv[8];
  dev::Triple res[16];
#pragma unroll
  for (int j = 0; j < 8; ++j) pj[j] = j < m ? p[c0 + j] : 0.f;
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    if (r < n) {
      const float sh = rh[r0 + r], sl = rl[r0 + r], sm = rm[r0 + r];
      res[r].h = sh;
      res[r].l = sl;
      res[r].m = sm;
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < m) res[r].fma(-J[j * n + r], pj[j]);
      if (!isfinite(res[r].h + res[r].l)) {
        double v = (double)sh + ((double)sl + (double)sm);
        for (int j = 0; j < m; ++j) v -= (double)J[j * n + r] * (double)p[c0 + j];
        res[r] = triple_of(v);
      }
      rh[r0 + r] = res[r].h;
      rl[r0 + r] = res[r].l;
      rm[r0 + r] = res[r].m;
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    hv[k] = 0.f;
    if (k < m) {
      dev::Triple g;
#pragma unroll
      for (int r = 0; r < 16; ++r)
        if (r < n) g.fma(J[k * n + r], res[r].h, res[r].l, res[r].m);
      double gv = g.value();
      if (!isfinite(gv)) {
        gv = 0.0;
#pragma unroll
        for (int r = 0; r < 16; ++r)
          if (r < n) gv += (double)J[k * n + r] * res[r].value();
      }
      const double d = O.D[c0 + k];
      float v = (float)(gv - lam * d * d * (double)pj[k]);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < k) v -= F[k * na + j] * hv[j];
      hv[k] = v / F[k * na + k];
      h[c0 + k] = hv[k];
    }
  }
}

// 3. shared columns, first part: S^T r per chunk of kSumRows rows.  A warp takes a column at a
// time; the chunk's r is in shared memory.
constexpr int kSumRows = 2048;
constexpr int kSumWarps = 8;
constexpr int kSumCols = 2;    // columns per warp

template <int V>
__global__ void __launch_bounds__(32 * kSumWarps) dense_cols_kernel(const float* S, int64_t rows, int s, const float* rh,
                                                                    const float* rl, const float* rm, double* part) {
  dev::chain_wait();
  __shared__ __align__(16) float rh_s[kSumRows], rl_s[kSumRows], rm_s[kSumRows];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t row0 = (int64_t)blockIdx.x * kSumRows;
  const int nr = (int)(rows - row0 < kSumRows ? rows - row0 : kSumRows);
  for (int e = threadIdx.x; e < nr; e += 32 * kSumWarps) {
    rh_s[e] = rh[row0 + e];
    rl_s[e] = rl[row0 + e];
    rm_s[e] = rm[row0 + e];
  }
  __syncthreads();
  for (int u = 0; u < kSumCols; ++u) {
    const int c = ((int)blockIdx.y * kSumCols + u) * kSumWarps + warp;
    if (c >= s) return;
    const float* src = S + (int64_t)c * rows + row0;
    dev::Triple sum;
#pragma unroll 4
    for (int e = lane * V; e < nr; e += 32 * V) {   // V divides nr
      Vec<V> a, h, l, m;
      a.load(src + e);
      h.load(rh_s + e);
      l.load(rl_s + e);
      m.load(rm_s + e);
#pragma unroll
      for (int q = 0; q < V; ++q) sum.fma(a.v[q], h.v[q], l.v[q], m.v[q]);
    }
    double t = sum.value();
    if (__any_sync(0xffffffffu, !isfinite(t))) {
      t = 0.0;
      for (int e = lane; e < nr; e += 32) t += (double)src[e] * ((double)rh_s[e] + ((double)rl_s[e] + (double)rm_s[e]));
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
    if (lane == 0) part[(int64_t)blockIdx.x * s + c] = t;
  }
}

// ... second part: R12^T h per chunk of kR12Rows rows of R12 (row-major, s values each).  A
// thread takes V adjacent columns; groups of threads take alternate rows.
constexpr int kR12Rows = 512;
constexpr int kR12Threads = 256;

template <int V>
__global__ void __launch_bounds__(kR12Threads) dense_r12_kernel(const float* R12, int64_t nb, int s, const float* h,
                                                                double* part) {
  dev::chain_wait();
  __shared__ float h_s[kR12Rows];
  __shared__ double sum_s[kR12Threads * V];
  const int64_t j0 = (int64_t)blockIdx.x * kR12Rows;
  const int nj = (int)(nb - j0 < kR12Rows ? nb - j0 : kR12Rows);
  const int units = s / V;                                   // V divides s
  const int u0 = (int)blockIdx.y * kR12Threads;
  const int nu = min(kR12Threads, units - u0);               // column units of this CTA
  const int groups = kR12Threads / nu;
  const int u = (int)threadIdx.x % nu, g = (int)threadIdx.x / nu;
  for (int e = threadIdx.x; e < nj; e += kR12Threads) h_s[e] = h[j0 + e];
  __syncthreads();
  if (g < groups) {
    dev::Triple sum[V];
    const float* src = R12 + j0 * s + (int64_t)(u0 + u) * V;
#pragma unroll 4
    for (int j = g; j < nj; j += groups) {
      Vec<V> a;
      a.load(src + (int64_t)j * s);
#pragma unroll
      for (int q = 0; q < V; ++q) sum[q].fma(a.v[q], h_s[j]);
    }
#pragma unroll
    for (int q = 0; q < V; ++q) {
      double t = sum[q].value();
      if (!isfinite(t)) {
        t = 0.0;
        for (int j = g; j < nj; j += groups) t += (double)src[(int64_t)j * s + q] * (double)h_s[j];
      }
      sum_s[(g * nu + u) * V + q] = t;
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < nu * V; c += kR12Threads) {
    double t = 0;
    for (int k = 0; k < groups; ++k) t += sum_s[k * nu * V + c];
    part[(int64_t)blockIdx.x * s + (int64_t)u0 * V + c] = t;
  }
}

// ... and their sum, one warp per column in a fixed order: g_S = S^T r - R12^T h - lambda D^2 p_S.
__global__ void __launch_bounds__(256) dense_gsum_kernel(const double* part_s, int64_t ns, const double* part_r,
                                                         int64_t nr, int s, const double* DS, const float* pS,
                                                         double lam, double* gS) {
  dev::chain_wait();
  const int c = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (c >= s) return;
  double t = 0;
  for (int64_t k = lane; k < ns; k += 32) t += part_s[k * s + c];
  for (int64_t k = lane; k < nr; k += 32) t -= part_r[k * s + c];
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
  if (lane == 0) {
    const double d = DS[c];
    gS[c] = t - lam * d * d * (double)pS[c];
  }
}

inline unsigned nblk(int64_t n, int64_t t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

#define DS_LAUNCH(ctx, ...)                         \
  do {                                              \
    __VA_ARGS__;                                    \
    (ctx)->launches += 1;                           \
    QRKIT_CUDA_TRY(ctx, cudaGetLastError());        \
  } while (0)

template <typename T>
qrkit_status dense_backsub(qrkit_ctx* ctx, bool chained, const T* R, int64_t ld, int s, const T* c, T* x) {
  DS_LAUNCH(ctx, launch_kernel(chained, ctx->stream, 1, tri_cta(s), 0, tri_backsub_kernel<T>, R, ld, s, c, x,
                               ctx->d_status));
  return QRKIT_OK;
}
template qrkit_status dense_backsub<float>(qrkit_ctx*, bool, const float*, int64_t, int, const float*, float*);
template qrkit_status dense_backsub<double>(qrkit_ctx*, bool, const double*, int64_t, int, const double*, double*);

template <typename T>
qrkit_status dense_normal(qrkit_ctx* ctx, const T* R, int64_t ld, int s, const double* g, T* dp, T* x) {
  DS_LAUNCH(ctx, chain_launch(ctx->stream, 1, tri_cta(s), 0, tri_normal_kernel<T>, R, ld, s, g, dp, x,
                              ctx->d_status));
  return QRKIT_OK;
}
template qrkit_status dense_normal<float>(qrkit_ctx*, const float*, int64_t, int, const double*, float*, float*);
template qrkit_status dense_normal<double>(qrkit_ctx*, const double*, int64_t, int, const double*, double*, double*);

// By warps a block's rows of R12 are read together, which hides latency while there are few blocks; but every lane
// repeats the substitution, and a sum over the warp costs five additions of all lanes.  A thread per block does
// neither: with many blocks its strided reads of R12 are covered by the other threads.  Doubles, where the warp pays
// the FP64 unit for each lane, cross at 9 to 22 blocks per SM (s = 16 .. 64), floats at 23 (s = 16, one column) to 260
// (s = 48, eight columns) along 16 + s m / 2; from s = 64 on, where float rows are read 16 bytes a lane, the warp is
// as fast or faster, one column per block and s = 64 apart.  The whole R solve with s = 30 and blocks of 5 x 3: 8,000
// in double 50 us by warps, 28 by threads; 50,000 in float 40 and 18; 1,000 in double 24 and 27; 4,000 in float 12
// and 15.
template <typename T>
static bool backsub_by_warps(const qrkit_ctx* ctx, int64_t K, int s) {
  if (sizeof(T) == 8) return K <= (int64_t)ctx->num_sms * (5 + s / 4);
  return s > 64 || (s == 64 && ctx->plan.max_m > 1) || K <= (int64_t)ctx->num_sms * (16 + s * ctx->plan.max_m / 2);
}

template <typename T>
qrkit_status dense_block_backsub(qrkit_ctx* ctx, bool chained, const ComposedView<T>& V, const FactorOut<T>& O,
                                 const T* rhs, const T* xS, T* x, int accumulate) {
  if (backsub_by_warps<T>(ctx, V.K, V.s))
    DS_LAUNCH(ctx, launch_kernel(chained, ctx->stream, nblk(V.K * 32, kWarpBackThreads), kWarpBackThreads, 0,
                                 block_backsub_warp_kernel<T>, V, O, rhs, xS, x, accumulate));
  else
    DS_LAUNCH(ctx, launch_kernel(chained, ctx->stream, nblk(V.K, kThreadBackThreads), kThreadBackThreads, 0,
                                 block_backsub_thread_kernel<T>, V, O, rhs, xS, x, accumulate));
  return QRKIT_OK;
}
template qrkit_status dense_block_backsub<float>(qrkit_ctx*, bool, const ComposedView<float>&, const FactorOut<float>&,
                                                 const float*, const float*, float*, int);
template qrkit_status dense_block_backsub<double>(qrkit_ctx*, bool, const ComposedView<double>&, const FactorOut<double>&,
                                                  const double*, const double*, double*, int);

size_t dense_refine_bytes(int64_t rows, int64_t nb, int s) {
  const int64_t chunks = (rows + kSumRows - 1) / kSumRows + (nb + kR12Rows - 1) / kR12Rows;
  return (size_t)chunks * s * sizeof(double) + 3 * (size_t)((rows + 3) & ~int64_t(3)) * sizeof(float);
}

qrkit_status dense_refine_gradient(qrkit_ctx* ctx, const ComposedView<float>& V, const FactorOut<float>& O,
                                   const float* b, const float* p, double lam, void* ws, float* h, double* gS) {
  cudaStream_t st = ctx->stream;
  const int s = V.s;
  const int64_t ns = (V.rows + kSumRows - 1) / kSumRows, nr = (V.nb + kR12Rows - 1) / kR12Rows;
  double* part_s = (double*)ws;
  double* part_r = part_s + ns * s;
  float* rh = (float*)(part_r + nr * s);
  float* rl = rh + ((V.rows + 3) & ~int64_t(3));
  float* rm = rl + ((V.rows + 3) & ~int64_t(3));
  // 16-byte loads where every column of the caller's S is 16-byte aligned
  const bool v4 = (V.rows & 3) == 0 && (reinterpret_cast<uintptr_t>(V.S) & 15) == 0;
  if (v4)
    DS_LAUNCH(ctx, chain_launch(st, nblk(V.rows, 128), 32 * kRowWarps, 0, dense_rows_kernel<4>, V.S, V.rows, s, b,
                                p + V.nb, rh, rl, rm));
  else
    DS_LAUNCH(ctx, chain_launch(st, nblk(V.rows, 32), 32 * kRowWarps, 0, dense_rows_kernel<1>, V.S, V.rows, s, b,
                                p + V.nb, rh, rl, rm));
  DS_LAUNCH(ctx, chain_launch(st, nblk(V.K, 128), 128, 0, dense_blocks_kernel, V, O, p, lam, rh, rl, rm, h));
  const dim3 gs((unsigned)ns, nblk(s, kSumWarps * kSumCols));
  if (v4)
    DS_LAUNCH(ctx, chain_launch(st, gs, 32 * kSumWarps, 0, dense_cols_kernel<4>, V.S, V.rows, s, rh, rl, rm, part_s));
  else
    DS_LAUNCH(ctx, chain_launch(st, gs, 32 * kSumWarps, 0, dense_cols_kernel<1>, V.S, V.rows, s, rh, rl, rm, part_s));
  if ((s & 3) == 0)
    DS_LAUNCH(ctx, chain_launch(st, dim3((unsigned)nr, nblk(s / 4, kR12Threads)), kR12Threads, 0, dense_r12_kernel<4>,
                                O.R12, V.nb, s, h, part_r));
  else
    DS_LAUNCH(ctx, chain_launch(st, dim3((unsigned)nr, nblk(s, kR12Threads)), kR12Threads, 0, dense_r12_kernel<1>,
                                O.R12, V.nb, s, h, part_r));
  DS_LAUNCH(ctx, chain_launch(st, nblk((int64_t)s * 32, 256), 256, 0, dense_gsum_kernel, part_s, ns, part_r, nr, s,
                              O.D + V.nb, p + V.nb, lam, gS));
  return QRKIT_OK;
}

}  // namespace qrkit
