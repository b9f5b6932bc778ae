// Column sums of a windowed S in plans whose blocks all have one shape (Sec. 4.2), and a refinement step's
// gradient with them (Sec. 5.1).
//
// A shared column's sum runs over the blocks whose windows hold it, which lie anywhere in memory.  The blocks
// sorted by window start (block_sort) bring those of one start together: eight lanes take kRun
// consecutive sorted blocks, lane t the window's column t, read the blocks' rows of S (a whole 64-byte
// window at a time for 2 x 1 blocks of floats) and keep the sum in registers, three floats, until the start changes.
// One atomic per column and run then, where a thread per block added its eight columns to shared
// memory by FP64 atomics: those retry as compare-and-swap loops around an FP64 add, and a warp's FP64
// instruction holds the SM's FP64 unit for 16 cycles (83 % busy).  10.5 million blocks 2 x 1, windows of
// 8: the gradient takes 870 us (residuals 273, sums 597) against 2.20 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include "chain.cuh"
#include "device_util.cuh"
#include "internal.h"
#include "sums.cuh"

namespace qrkit {
namespace {

constexpr int kLanes = 8;     // lanes of a run: the widest window
constexpr int kRun = 32;      // sorted blocks of a run
constexpr int kThreads = 256;

// Sums over a block's rows: float pairs for blocks up to 6 x 2 of floats, three floats for larger ones, doubles for doubles;
// a residual is kept as such a sum.
struct DoubleSum {
  double s = 0.0;
  __device__ __forceinline__ void fma(double a, double x) { s += a * x; }
  __device__ __forceinline__ double value() const { return s; }
};
template <typename T, int NR>
struct BlockSum;
template <int NR>
struct BlockSum<double, NR> {
  static constexpr int kValues = 1;
  DoubleSum s;
  __device__ __forceinline__ void start(double b) { s.s = b; }
  __device__ __forceinline__ void fma(double a, double x) { s.fma(a, x); }
  __device__ __forceinline__ void fma(double a, const double (&x)[1]) { s.fma(a, x[0]); }
  __device__ __forceinline__ void get(double (&v)[1]) const { v[0] = s.s; }
  __device__ __forceinline__ double value() const { return s.s; }
};
template <int NR>
struct BlockSum<float, NR> {
  static constexpr int kValues = NR > 6 ? 3 : 2;
  dev::Triple s;   // of a pair, two of the three
  __device__ __forceinline__ void start(float b) { s.h = b; }
  __device__ __forceinline__ void fma(float a, float x) {
    if constexpr (kValues == 3) {
      s.fma(a, x);
    } else {
      dev::Pair p;
      p.h = s.h;
      p.l = s.l;
      p.fma(a, x);
      s.h = p.h;
      s.l = p.l;
    }
  }
  __device__ __forceinline__ void fma(float a, const float (&x)[kValues]) {
    if constexpr (kValues == 3) {
      s.fma(a, x[0], x[1], x[2]);
    } else {
      fma(a, x[0]);
      s.l = __fmaf_rn(a, x[1], s.l);
    }
  }
  __device__ __forceinline__ void get(float (&v)[kValues]) const {
    v[0] = s.h;
    v[1] = s.l;
    if constexpr (kValues == 3) v[2] = s.m;
  }
  __device__ __forceinline__ double value() const { return s.value(); }
  __device__ __forceinline__ void set(double v) {
    s.h = (float)v;
    s.l = (float)(v - (double)s.h);
    s.m = (float)(v - (double)s.h - (double)s.l);
  }
};

// What a lane of a run adds up over its blocks: products (kGrad), or squares; no less accurate than in double.
template <typename T, bool kGrad>
struct RunSum {
  DoubleSum s;
  __device__ __forceinline__ void fma(T a, T x) { s.fma(a, x); }
  __device__ __forceinline__ void fma(T a, const T (&x)[1]) { s.fma(a, x[0]); }
  template <int N>
  __device__ __forceinline__ void squares(const T (&x)[N]) {
#pragma unroll
    for (int r = 0; r < N; ++r) s.fma(x[r], x[r]);
  }
  __device__ __forceinline__ double value() const { return s.value(); }
};
template <>
struct RunSum<float, true> {
  dev::Triple s;
  __device__ __forceinline__ void fma(float a, float x) { s.fma(a, x); }
  __device__ __forceinline__ void fma(float a, const float (&x)[3]) { s.fma(a, x[0], x[1], x[2]); }
  // a small block's products (residuals of two floats; zeros past its rows and columns) as a pair of its own, then added
  template <int NR, int MM>
  __device__ __forceinline__ void block(const float (&a)[NR], const float (&x)[NR][2], const float (&b)[MM],
                                        const float (&y)[MM]) {
    dev::Pair p;
    p.h = __fmul_rn(a[0], x[0][0]);
    p.l = __fmaf_rn(a[0], x[0][1], __fmaf_rn(a[0], x[0][0], -p.h));
#pragma unroll
    for (int r = 1; r < NR; ++r) {
      const float q = __fmul_rn(a[r], x[r][0]);
      p.add(q, __fmaf_rn(a[r], x[r][1], __fmaf_rn(a[r], x[r][0], -q)));
    }
#pragma unroll
    for (int k = 0; k < MM; ++k) p.fma(b[k], y[k]);
    s.add(p.h);
    s.low(p.l);
  }
  __device__ __forceinline__ double value() const { return s.value(); }
};
template <>
struct RunSum<float, false> {
  dev::Squares s;
  template <int N>
  __device__ __forceinline__ void squares(const float (&x)[N]) {
    s.add(x);
  }
  __device__ __forceinline__ double value() const { return s.value(); }
};

// Eight lanes per run of kRun sorted blocks.  kGrad: sum of S^T r - R12^T h; else of the squares of S.
template <typename T, bool kGrad, int NR, int MM>
__global__ void __launch_bounds__(kThreads) window_sums_kernel(WindowSums<T> A) {
  dev::chain_wait();
  const int64_t run = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / kLanes;
  const int t = threadIdx.x % kLanes;
  const int64_t p0 = run * kRun, p1 = p0 + kRun < A.K ? p0 + kRun : A.K;
  if (p0 >= A.K || t >= A.w) return;
  const int n = A.n, m = A.m, w = A.w;
  constexpr int RV = BlockSum<T, NR>::kValues;
  RunSum<T, kGrad> acc;
  int64_t cur = -1, first = p0;   // start of the blocks added up, and the first of them
  auto flush = [&](int64_t end) {
    if (cur >= 0 && cur + t < A.s) {
      double v = acc.value();
      if (kGrad && sizeof(T) == 4 && !isfinite(v)) {   // a product left the float range: these blocks again in double
        v = 0.0;
        for (int64_t q = first; q < end; ++q) {
          const int64_t i = A.bord[q];
          for (int r = 0; r < n; ++r) {
            double x = 0.0;
            for (int e = RV - 1; e >= 0; --e) x += (double)A.r[RV * (i * n + r) + e];
            v += (double)A.S[(i * w + t) * n + r] * x;
          }
          for (int k = 0; k < m; ++k) v -= (double)A.R12[(i * m + k) * w + t] * (double)A.h[i * m + k];
        }
      }
      if (v != 0.0) atomicAdd(A.out + cur + t, v);
    }
    acc = RunSum<T, kGrad>();
    first = end;
  };
  constexpr int U = NR * MM <= 2 ? 4 : 1;   // blocks whose loads are in flight together
  for (int64_t q0 = p0; q0 < p1; q0 += U) {
    int64_t i[U];
    int32_t st[U];
    T sv[U][NR], res[U][NR][RV], rv[U][MM], hv[U][MM];
#pragma unroll
    for (int u = 0; u < U; ++u) i[u] = q0 + u < p1 ? A.bord[q0 + u] : -1;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      st[u] = 0;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        sv[u][r] = T(0);
#pragma unroll
        for (int e = 0; e < RV; ++e) res[u][r][e] = T(0);
      }
#pragma unroll
      for (int k = 0; k < MM; ++k) rv[u][k] = hv[u][k] = T(0);
      if (i[u] < 0) continue;
      st[u] = A.start[i[u]];
      const T* S = A.S + (i[u] * w + t) * n;   // block i: n x w column-major
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (r < n) sv[u][r] = S[r];
      if constexpr (kGrad) {
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (r < n) {
#pragma unroll
            for (int e = 0; e < RV; ++e) res[u][r][e] = A.r[RV * (i[u] * n + r) + e];
          }
#pragma unroll
        for (int k = 0; k < MM; ++k)
          if (k < m) {
            rv[u][k] = A.R12[(i[u] * m + k) * w + t];
            hv[u][k] = -A.h[i[u] * m + k];
          }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (i[u] < 0) continue;
      if (st[u] != cur) {
        flush(q0 + u);
        cur = st[u];
      }
      if constexpr (!kGrad) acc.squares(sv[u]);   // zeros past row n
      if constexpr (kGrad && RV == 2) {
        acc.block(sv[u], res[u], rv[u], hv[u]);
      } else if constexpr (kGrad) {
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (r < n) acc.fma(sv[u][r], res[u][r]);
#pragma unroll
        for (int k = 0; k < MM; ++k)
          if (k < m) acc.fma(rv[u][k], hv[u][k]);
      }
    }
  }
  flush(p1);
}

// A block per thread: r = b - J p - S p_S, g_B = J^T r - lambda D^2 p, h_B = R_i^{-T} g_B.
template <typename T, int NR, int MM>
__global__ void __launch_bounds__(128) window_blocks_kernel(ComposedView<T> V, FactorOut<T> O, const T* b, const T* p,
                                                            double lam, int n, int m, T* r, T* h) {
  dev::chain_wait();
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (i >= V.K) return;
  const int na = n + (O.damp ? m : 0), w = V.w;
  const int64_t c0 = i * m, r0 = i * n;
  const T* J = V.J + i * n * m;
  const T* S = V.S + r0 * w;
  const T* F = O.Fa + O.aug_off[i];
  const int64_t st = V.start[i];
  T pj[MM], ps[kLanes];
#pragma unroll
  for (int j = 0; j < MM; ++j) pj[j] = j < m ? -p[c0 + j] : T(0);
#pragma unroll
  for (int t = 0; t < kLanes; ++t) ps[t] = t < w && st + t < V.s ? -p[V.nb + st + t] : T(0);
  using Res = BlockSum<T, NR>;
  constexpr int RV = Res::kValues;
  Res res[NR];
  bool done = false;
  if constexpr (sizeof(T) == 4 && NR == 2) {
    if (w == 8 && n == 2 && (reinterpret_cast<uintptr_t>(V.S) & 15) == 0) {   // the window by 16-byte loads
      const float4* s4 = reinterpret_cast<const float4*>(S);
#pragma unroll
      for (int q = 0; q < 2; ++q) res[q].start(b[r0 + q]);
#pragma unroll
      for (int q = 0; q < 2; ++q) res[q].fma(J[q], pj[0]);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 v = s4[q];
        res[0].fma(v.x, ps[2 * q]);
        res[1].fma(v.y, ps[2 * q]);
        res[0].fma(v.z, ps[2 * q + 1]);
        res[1].fma(v.w, ps[2 * q + 1]);
      }
      done = true;
    }
  }
  if (!done) {
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      if (q < n) {
        res[q].start(b[r0 + q]);
#pragma unroll
        for (int j = 0; j < MM; ++j)
          if (j < m) res[q].fma(J[j * n + q], pj[j]);
#pragma unroll
        for (int t = 0; t < kLanes; ++t)
          if (t < w) res[q].fma(S[t * n + q], ps[t]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NR; ++q)
    if (q < n) {
      if constexpr (RV == 3) {
        if (!isfinite(res[q].s.h + res[q].s.l)) {   // a product left the float range
          double v = (double)b[r0 + q];
          for (int j = 0; j < m; ++j) v -= (double)J[j * n + q] * (double)p[c0 + j];
          for (int t = 0; t < w; ++t)
            if (st + t < V.s) v -= (double)S[t * n + q] * (double)p[V.nb + st + t];
          res[q].set(v);
        }
      }
      T v[RV];
      res[q].get(v);
#pragma unroll
      for (int e = 0; e < RV; ++e) r[RV * (r0 + q) + e] = v[e];
    }
  T hv[MM];
#pragma unroll
  for (int k = 0; k < MM; ++k) {
    hv[k] = T(0);
    if (k < m) {
      Res g;
#pragma unroll
      for (int q = 0; q < NR; ++q)
        if (q < n) {
          T x[RV];
          res[q].get(x);
          g.fma(J[k * n + q], x);
        }
      double gv = g.value();
      if constexpr (RV == 3) {
        if (!isfinite(gv)) {
          gv = 0.0;
#pragma unroll
          for (int q = 0; q < NR; ++q)
            if (q < n) gv += (double)J[k * n + q] * res[q].value();
        }
      }
      const double d = O.D[c0 + k];
      T v = (T)(gv + lam * d * d * (double)pj[k]);
#pragma unroll
      for (int j = 0; j < MM; ++j)
        if (j < k) v -= F[k * na + j] * hv[j];
      hv[k] = v / F[k * na + k];
      h[c0 + k] = hv[k];
    }
  }
}

// ---- 2 x 1 blocks with windows of 8, one thread each: factorization, Q^T b and back-substitution ----
//
// The general small-block kernels read six tables of offsets per block and touch a window entry by entry (a warp's
// load spreads over 32 windows).  A plan of one shape needs no offsets, and rows of a window are whole 16-byte pieces:
// 10.5 million blocks: factorization 634 -> 354 us, Q^T b 135 -> 105 us, back-substitution 140 -> 106 us.
// The arithmetic is that of the general kernels.
template <typename T, int N>
__device__ __forceinline__ void load_wide(T (&v)[N], const T* src) {   // src 16-byte aligned
  constexpr int E = 16 / (int)sizeof(T);
  union Piece {
    uint4 q;
    T t[E];
  };
#pragma unroll
  for (int k = 0; k < N / E; ++k) {
    Piece p;
    p.q = reinterpret_cast<const uint4*>(src)[k];
#pragma unroll
    for (int e = 0; e < E; ++e) v[k * E + e] = p.t[e];
  }
}
template <typename T, int N>
__device__ __forceinline__ void store_wide(T* dst, const T (&v)[N]) {   // dst 16-byte aligned
  constexpr int E = 16 / (int)sizeof(T);
  union Piece {
    uint4 q;
    T t[E];
  };
#pragma unroll
  for (int k = 0; k < N / E; ++k) {
    Piece p;
#pragma unroll
    for (int e = 0; e < E; ++e) p.t[e] = v[k * E + e];
    reinterpret_cast<uint4*>(dst)[k] = p.q;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) window21_factor_kernel(ComposedView<T> V, FactorOut<T> O) {
  dev::chain_wait();
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= V.K) return;
  const int64_t at = (int64_t)O.bpos[i] * O.q;   // the block's first reduced row
  T S[16];
  load_wide(S, V.S + 16 * i);
  const T alpha = V.J[2 * i];
  T b1 = V.J[2 * i + 1], b2 = O.damp ? (T)(O.lam_half * O.D[i]) : T(0);
  T sq = b1 * b1;
  if (O.damp) sq += b2 * b2;
  const T norm = sqrt(alpha * alpha + sq);
  T beta = 0, tau = 0, scale = 0;
  if (norm != T(0)) {
    beta = alpha >= T(0) ? -norm : norm;
    tau = (beta - alpha) / beta;
    scale = T(1) / (alpha - beta);
  } else if (O.status) {
    atomicCAS(O.status, 0, QRKIT_ESINGULAR);
  }
  b1 *= scale;
  b2 *= scale;
  const int na = O.damp ? 3 : 2;
  T* F = O.Fa + na * i;
  F[0] = beta;
  F[1] = b1;
  if (O.damp) F[2] = b2;
  O.tau[i] = tau;
  T r12[8], x0[8], x1[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const T w = (S[2 * c] + b1 * S[2 * c + 1]) * tau;
    r12[c] = S[2 * c] - w;
    x0[c] = S[2 * c + 1] - w * b1;
    x1[c] = T(0) - w * b2;
  }
  store_wide(O.R12 + 8 * i, r12);
  store_wide(O.Xw + 8 * at, x0);
  if (O.damp) store_wide(O.Xw + 8 * (at + 1), x1);
}

template <typename T>
__global__ void __launch_bounds__(256) window21_qt_kernel(ComposedView<T> V, FactorOut<T> O, const T* b, T* rhs0) {
  dev::chain_wait();
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= V.K) return;
  const int64_t at = (int64_t)O.bpos[i] * O.q;
  const T y0 = b[2 * i], y1 = b[2 * i + 1];
  const T* F = O.Fa + (O.damp ? 3 : 2) * i;
  const T b1 = F[1], b2 = O.damp ? F[2] : T(0);
  const T w = (y0 + b1 * y1) * O.tau[i];
  O.ctop[i] = y0 - w;
  if (!rhs0) return;
  rhs0[at] = y1 - w * b1;
  if (O.damp) rhs0[at + 1] = T(0) - w * b2;
}

template <typename T>
__global__ void __launch_bounds__(256) window21_backsub_kernel(ComposedView<T> V, FactorOut<T> O, const T* rhs,
                                                               const T* xS, T* x, int accumulate) {
  dev::chain_wait();
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= V.K) return;
  T y = rhs[i];
  if (xS) {
    const int64_t st = V.start[i];
    T r12[8];
    load_wide(r12, O.R12 + 8 * i);
#pragma unroll
    for (int t = 0; t < 8; ++t)
      if (st + t < V.s) y -= r12[t] * xS[st + t];
  }
  y = y / O.Fa[(O.damp ? 3 : 2) * i];
  x[i] = accumulate ? x[i] + y : y;
}

inline unsigned nblk(int64_t n, int64_t t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// A kernel template KERNEL<.., NR, MM> in the instantiation that holds blocks n x m.
#define WS_SHAPED(ctx, n, m, LAUNCH21, LAUNCH62, LAUNCH168) \
  do {                                                      \
    if ((m) == 1 && (n) <= 2) LAUNCH21;                     \
    else if ((m) <= 2 && (n) <= 6) LAUNCH62;                \
    else LAUNCH168;                                         \
    (ctx)->launches += 1;                                   \
    QRKIT_CUDA_TRY(ctx, cudaGetLastError());                \
  } while (0)

template <typename T>
qrkit_status window_square_sums(qrkit_ctx* ctx, const WindowSums<T>& A) {
  const unsigned g = nblk((A.K + kRun - 1) / kRun * kLanes, kThreads);
  WS_SHAPED(ctx, A.n, A.m, (chain_launch(ctx->stream, g, kThreads, 0, (window_sums_kernel<T, false, 2, 1>), A)),
            (chain_launch(ctx->stream, g, kThreads, 0, (window_sums_kernel<T, false, 6, 2>), A)),
            (chain_launch(ctx->stream, g, kThreads, 0, (window_sums_kernel<T, false, 16, 8>), A)));
  return QRKIT_OK;
}
template qrkit_status window_square_sums<float>(qrkit_ctx*, const WindowSums<float>&);
template qrkit_status window_square_sums<double>(qrkit_ctx*, const WindowSums<double>&);

template <typename T>
qrkit_status window_refine_gradient(qrkit_ctx* ctx, const ComposedView<T>& V, const FactorOut<T>& O, const T* b,
                                    const T* p, double lam, const WindowSums<T>& A) {
  const unsigned gb = nblk(V.K, 128), g = nblk((A.K + kRun - 1) / kRun * kLanes, kThreads);
  T* r = const_cast<T*>(A.r);
  T* h = const_cast<T*>(A.h);
  WS_SHAPED(ctx, A.n, A.m, (chain_launch(ctx->stream, gb, 128, 0, (window_blocks_kernel<T, 2, 1>), V, O, b, p, lam,
                                         A.n, A.m, r, h)),
            (chain_launch(ctx->stream, gb, 128, 0, (window_blocks_kernel<T, 6, 2>), V, O, b, p, lam, A.n, A.m, r, h)),
            (chain_launch(ctx->stream, gb, 128, 0, (window_blocks_kernel<T, 16, 8>), V, O, b, p, lam, A.n, A.m, r,
                          h)));
  WS_SHAPED(ctx, A.n, A.m, (chain_launch(ctx->stream, g, kThreads, 0, (window_sums_kernel<T, true, 2, 1>), A)),
            (chain_launch(ctx->stream, g, kThreads, 0, (window_sums_kernel<T, true, 6, 2>), A)),
            (chain_launch(ctx->stream, g, kThreads, 0, (window_sums_kernel<T, true, 16, 8>), A)));
  return QRKIT_OK;
}
template qrkit_status window_refine_gradient<float>(qrkit_ctx*, const ComposedView<float>&, const FactorOut<float>&,
                                                    const float*, const float*, double, const WindowSums<float>&);
template qrkit_status window_refine_gradient<double>(qrkit_ctx*, const ComposedView<double>&, const FactorOut<double>&,
                                                     const double*, const double*, double, const WindowSums<double>&);

bool window21(const qrkit_ctx* ctx) {
  const Plan& P = ctx->plan;
  return ctx->comp.bins && P.max_n == 2 && P.max_m == 1 && ctx->plan.s.window == 8;
}

template <typename T>
qrkit_status window21_factor(qrkit_ctx* ctx, const ComposedView<T>& V, const FactorOut<T>& O) {
  QRKIT_CUDA_TRY(ctx, chain_launch(ctx->stream, nblk(V.K, 256), 256, 0, window21_factor_kernel<T>, V, O));
  ctx->launches += 1;
  return QRKIT_OK;
}
template <typename T>
qrkit_status window21_qt(qrkit_ctx* ctx, bool chained, const ComposedView<T>& V, const FactorOut<T>& O, const T* b,
                         T* rhs0) {
  QRKIT_CUDA_TRY(ctx, launch_kernel(chained, ctx->stream, nblk(V.K, 256), 256, 0, window21_qt_kernel<T>, V, O, b, rhs0));
  ctx->launches += 1;
  return QRKIT_OK;
}
template <typename T>
qrkit_status window21_backsub(qrkit_ctx* ctx, const ComposedView<T>& V, const FactorOut<T>& O, const T* rhs, const T* xS,
                              T* x, int accumulate) {
  QRKIT_CUDA_TRY(ctx, chain_launch(ctx->stream, nblk(V.K, 256), 256, 0, window21_backsub_kernel<T>, V, O, rhs, xS, x,
                                   accumulate));
  ctx->launches += 1;
  return QRKIT_OK;
}
#define WINDOW21_TYPES(T)                                                                                          \
  template qrkit_status window21_factor<T>(qrkit_ctx*, const ComposedView<T>&, const FactorOut<T>&);              \
  template qrkit_status window21_qt<T>(qrkit_ctx*, bool, const ComposedView<T>&, const FactorOut<T>&, const T*, T*); \
  template qrkit_status window21_backsub<T>(qrkit_ctx*, const ComposedView<T>&, const FactorOut<T>&, const T*,    \
                                            const T*, T*, int);
WINDOW21_TYPES(float)
WINDOW21_TYPES(double)
#undef WINDOW21_TYPES

}  // namespace qrkit
