// Composed QR of the damped block-angular system (Sec. 4.1, 4.2, 4.5, 5.1, 5.2):
//   P_r [J; lambda^(1/2) D] = [[blkdiag(B_i), C], [0, lambda^(1/2) D_S]],
//   B_i = [J_i; lambda^(1/2) D_i], C_i = [S_i; 0]  (row interleave, Sec. 4.5 / 5.2).
// Steps: D = column norms (Sec. 5.2); per block Q_i R_i = qr(B_i) (Sec. 4.1) with Q_i^T
// applied to C_i (Sec. 4.2): top rows -> R12_i, bottom rows -> reduced shared block; the
// reduced block [stacked bottoms; lambda^(1/2) D_S] is factored by TSQR (tall-skinny QR:
// row tiles factored in parallel, their R's stacked and factored again); solve R p = Q^T b
// by back-substitution (Sec. 5.1); optional refinement with FP64 residuals.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "chain.cuh"
#include "device_util.cuh"
#include "internal.h"
#include "sums.cuh"

namespace qrkit {
namespace {

constexpr int kMaxRows = 16;   // augmented rows per block
constexpr int kMaxCols = 8;    // columns per block
constexpr int kChunk = 8;      // coupled columns processed per pass

__device__ __forceinline__ void record(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// ---- column norms D = diag(J^T J)^(1/2) (Sec. 5.2): sums in double, those of a float dense S as
// sums of three floats per thread first (FP64 runs at 1/73 of the FP32 rate: 811 us in FP64 for an S of
// 819 MB, 237 us so) ----
template <typename T>
__global__ void colnorm_blocks_kernel(ComposedView<T> V, double* sq) {
  dev::chain_wait();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= V.K) return;
  const int n = V.n[i], m = V.m[i];
  const T* J = V.J + V.val_off[i];
  for (int j = 0; j < m; ++j) {
    double s = 0;
    for (int r = 0; r < n; ++r) {
      const double x = (double)J[j * n + r];
      s += x * x;
    }
    sq[V.col_off[i] + j] = s;
  }
}

// Dense S (column-major, ld = rows of J): squared column norms in two deterministic passes.
// Pass 1, one CTA per (chunk of kNormRows rows, shared column): strided per-thread sums, then
// the warps' sums in warp order; pass 2, one thread per column adds its chunks in order.
constexpr int kNormRows = 8192;
constexpr int kNormThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kNormThreads) colnorm_dense_part_kernel(ComposedView<T> V, double* part,
                                                                          int64_t nchunk) {
  dev::chain_wait();
  __shared__ double ws[kNormThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * kNormRows;
  const int64_t r1 = r0 + kNormRows < V.rows ? r0 + kNormRows : V.rows;
  for (int64_t col = blockIdx.y; col < V.s; col += gridDim.y) {
    const T* c = V.S + col * V.rows;
    double s = 0;
    if constexpr (sizeof(T) == sizeof(float)) {
      dev::Squares sum;
      for (int64_t r = r0 + threadIdx.x; r < r1; r += 8 * kNormThreads) {
        float x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = r + q * kNormThreads < r1 ? c[r + q * kNormThreads] : 0.f;
        sum.add(x);
      }
      s = sum.value();
    } else {
      for (int64_t r = r0 + threadIdx.x; r < r1; r += kNormThreads) {
        const double x = (double)c[r];
        s += x * x;
      }
    }
    for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (lane == 0) ws[wid] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0;
      for (int w = 0; w < kNormThreads / 32; ++w) t += ws[w];
      part[col * nchunk + blockIdx.x] = t;
    }
    __syncthreads();   // ws is reused by the next column
  }
}

__global__ void colnorm_dense_sum_kernel(const double* part, int64_t nchunk, int64_t s, double* sq) {
  dev::chain_wait();
  const int64_t col = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (col >= s) return;
  double t = 0;
  for (int64_t k = 0; k < nchunk; ++k) t += part[col * nchunk + k];
  sq[col] = t;
}

template <typename T>
__global__ void colnorm_window_kernel(ComposedView<T> V, double* sq) {
  dev::chain_wait();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= V.K) return;
  const int n = V.n[i];
  const T* C = V.S + V.row_off[i] * V.w;   // block i: n x w column-major
  for (int t = 0; t < V.w; ++t) {
    double s = 0;
    for (int r = 0; r < n; ++r) {
      const double x = (double)C[t * n + r];
      s += x * x;
    }
    const int64_t col = V.start[i] + t;
    if (s != 0.0 && col < V.s) atomicAdd(&sq[V.nb + col], s);
  }
}

__global__ void finalize_norms_kernel(const double* sq, double* D, int64_t N) {
  dev::chain_wait();
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= N) return;
  const double d = sqrt(sq[j]);
  D[j] = d == 0.0 ? 1.0 : d;   // zero column norm -> 1 (MINPACK convention)
}

// ---- per-block factor (Sec. 4.1) with Q_i^T applied to the coupled columns of windows (Sec. 4.2) ----
// One thread per block; the augmented block B_i = [J_i; lambda^(1/2) D_i] (na x m) is held
// column-major in local arrays.  Outputs: factor Fa (na x m, V below / R on and above the
// diagonal), tau, R12 rows (m x w) and the reduced rows (na - m rows).
// Small blocks (at most NA augmented rows and MM columns, e.g. the 2 x 1 blocks of curve and
// ellipse fits): the same factorization as the general path below, with every loop unrolled to
// the compile-time bounds (runtime sizes as guards), so the block, its reflectors and a chunk
// of coupled columns stay in registers instead of local memory.
template <typename T, int NA, int MM>
__device__ __forceinline__ void block_factor_small(const ComposedView<T>& V, const FactorOut<T>& O, int64_t i, int n,
                                                   int m) {
  const int na = n + (O.damp ? m : 0);
  const T* J = V.J + V.val_off[i];
  T B[MM][NA];
#pragma unroll
  for (int j = 0; j < MM; ++j)
#pragma unroll
    for (int r = 0; r < NA; ++r) {
      T v = T(0);
      if (j < m) {
        if (r < n) v = J[j * n + r];
        else if (O.damp && r - n == j) v = (T)(O.lam_half * O.D[V.col_off[i] + j]);
      }
      B[j][r] = v;
    }
  T tau[MM];
  bool bad = false;
#pragma unroll
  for (int k = 0; k < MM; ++k) {
    tau[k] = T(0);
    if (k < m) {
      T sq = 0;
#pragma unroll
      for (int r = 0; r < NA; ++r)
        if (r > k && r < na) sq += B[k][r] * B[k][r];
      const T alpha = B[k][k];
      const T norm = sqrt(alpha * alpha + sq);
      T beta = 0, t = 0, scale = 0;
      if (norm != T(0)) {
        beta = alpha >= T(0) ? -norm : norm;
        t = (beta - alpha) / beta;
        scale = T(1) / (alpha - beta);
      } else {
        bad = true;
      }
#pragma unroll
      for (int r = 0; r < NA; ++r)
        if (r > k) B[k][r] *= scale;
      B[k][k] = beta;
      tau[k] = t;
#pragma unroll
      for (int j = k + 1; j < MM; ++j) {
        if (j < m) {
          T w = B[j][k];
#pragma unroll
          for (int r = 0; r < NA; ++r)
            if (r > k && r < na) w += B[k][r] * B[j][r];
          w *= t;
          B[j][k] -= w;
#pragma unroll
          for (int r = 0; r < NA; ++r)
            if (r > k && r < na) B[j][r] -= w * B[k][r];
        }
      }
    }
  }
  if (bad) record(O.status, QRKIT_ESINGULAR);
  T* F = O.Fa + O.aug_off[i];
#pragma unroll
  for (int j = 0; j < MM; ++j)
#pragma unroll
    for (int r = 0; r < NA; ++r)
      if (j < m && r < na) F[j * na + r] = B[j][r];
#pragma unroll
  for (int k = 0; k < MM; ++k)
    if (k < m) O.tau[V.col_off[i] + k] = tau[k];
  if (V.coupled != QRKIT_COUPLED_WINDOW) return;   // a dense S: dense_block.cu
  const int64_t red0 = O.bpos ? (int64_t)O.bpos[i] * O.q : O.red_off[i];
  if constexpr (sizeof(T) == 4 && NA == 3 && MM == 1) {
    // the 2 x 1 point blocks of curve fits with windows of 8 (damped): the window, R12 and
    // the two reduced rows are moved by 16-byte loads and stores (all 32-byte aligned)
    if (V.coupled == QRKIT_COUPLED_WINDOW && V.w == 8 && n == 2 && m == 1 && na == 3 &&
        (reinterpret_cast<uintptr_t>(V.S) & 15) == 0) {   // the caller's S 16-byte aligned
      const float4* src = reinterpret_cast<const float4*>(V.S + V.row_off[i] * 8);   // 2 x 8 column-major
      float sv[16];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 v = src[q];
        sv[4 * q] = v.x;
        sv[4 * q + 1] = v.y;
        sv[4 * q + 2] = v.z;
        sv[4 * q + 3] = v.w;
      }
      float r12[8], x1[8], x2[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        // column c of the augmented window: rows (S[0][c], S[1][c], 0); reflector k = 0
        const float y0 = sv[2 * c], y1 = sv[2 * c + 1];
        float w = y0 + B[0][1] * y1;   // row 2 of the column is 0
        w *= tau[0];
        r12[c] = y0 - w;
        x1[c] = y1 - w * B[0][1];
        x2[c] = -w * B[0][2];
      }
      float4* dr = reinterpret_cast<float4*>(O.R12 + V.col_off[i] * 8);
      dr[0] = make_float4(r12[0], r12[1], r12[2], r12[3]);
      dr[1] = make_float4(r12[4], r12[5], r12[6], r12[7]);
      float4* dx = reinterpret_cast<float4*>(O.Xw + red0 * 8);
      dx[0] = make_float4(x1[0], x1[1], x1[2], x1[3]);
      dx[1] = make_float4(x1[4], x1[5], x1[6], x1[7]);
      dx[2] = make_float4(x2[0], x2[1], x2[2], x2[3]);
      dx[3] = make_float4(x2[4], x2[5], x2[6], x2[7]);
      if (O.Xstart) O.Xstart[red0] = O.Xstart[red0 + 1] = V.start[i];
      return;
    }
  }
  for (int c0 = 0; c0 < V.w; c0 += kChunk) {
    const int cw = min(kChunk, V.w - c0);
    T C[kChunk][NA];
#pragma unroll
    for (int c = 0; c < kChunk; ++c)
#pragma unroll
      for (int r = 0; r < NA; ++r) {
        T v = T(0);
        if (c < cw && r < n) v = V.S[V.row_off[i] * V.w + (int64_t)(c0 + c) * n + r];
        C[c][r] = v;
      }
#pragma unroll
    for (int k = 0; k < MM; ++k) {
      if (k < m) {
#pragma unroll
        for (int c = 0; c < kChunk; ++c) {
          T w = C[c][k];
#pragma unroll
          for (int r = 0; r < NA; ++r)
            if (r > k && r < na) w += B[k][r] * C[c][r];
          w *= tau[k];
          C[c][k] -= w;
#pragma unroll
          for (int r = 0; r < NA; ++r)
            if (r > k && r < na) C[c][r] -= w * B[k][r];
        }
      }
    }
#pragma unroll
    for (int c = 0; c < kChunk; ++c) {
      if (c < cw) {
#pragma unroll
        for (int r = 0; r < NA; ++r) {
          if (r < m) {
            O.R12[(V.col_off[i] + r) * (int64_t)V.w + c0 + c] = C[c][r];
          } else if (r < na) {
            const int64_t row = red0 + (r - m);
            O.Xw[row * V.w + c0 + c] = C[c][r];
            if (c0 + c == 0 && O.Xstart) O.Xstart[row] = V.start[i];
          }
        }
      }
    }
  }
}

// Plans whose blocks all fit (NA, MM) run this kernel (its register needs are those of the
// small blocks only).
template <typename T, int NA, int MM>
__global__ void block_factor_small_kernel(ComposedView<T> V, FactorOut<T> O) {
  dev::chain_wait();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= V.K) return;
  block_factor_small<T, NA, MM>(V, O, i, V.n[i], V.m[i]);
}

template <typename T>
__global__ void block_factor_kernel(ComposedView<T> V, FactorOut<T> O) {
  dev::chain_wait();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= V.K) return;
  const int n = V.n[i], m = V.m[i];
  const int na = n + (O.damp ? m : 0);
  T B[kMaxRows * kMaxCols];
  const T* J = V.J + V.val_off[i];
  for (int j = 0; j < m; ++j) {
    for (int r = 0; r < n; ++r) B[j * na + r] = J[j * n + r];
    if (O.damp)
      for (int r = 0; r < m; ++r)
        B[j * na + n + r] = (r == j) ? (T)(O.lam_half * O.D[V.col_off[i] + j]) : T(0);
  }
  T tau[kMaxCols];
  bool bad = false;
  for (int k = 0; k < m; ++k) {
    T* x = B + k * na;
    T sq = 0;
    for (int r = k + 1; r < na; ++r) sq += x[r] * x[r];
    const T alpha = x[k];
    const T norm = sqrt(alpha * alpha + sq);
    T beta = 0, t = 0, scale = 0;
    if (norm != T(0)) {
      beta = alpha >= T(0) ? -norm : norm;
      t = (beta - alpha) / beta;
      scale = T(1) / (alpha - beta);
    } else {
      bad = true;
    }
    for (int r = k + 1; r < na; ++r) x[r] *= scale;
    x[k] = beta;
    tau[k] = t;
    for (int j = k + 1; j < m; ++j) {
      T* y = B + j * na;
      T w = y[k];
      for (int r = k + 1; r < na; ++r) w += x[r] * y[r];
      w *= t;
      y[k] -= w;
      for (int r = k + 1; r < na; ++r) y[r] -= w * x[r];
    }
  }
  if (bad) record(O.status, QRKIT_ESINGULAR);
  T* F = O.Fa + O.aug_off[i];
  for (int e = 0; e < na * m; ++e) F[e] = B[e];
  for (int k = 0; k < m; ++k) O.tau[V.col_off[i] + k] = tau[k];
  // coupled columns, kChunk at a time
  if (V.coupled != QRKIT_COUPLED_WINDOW) return;   // a dense S: dense_block.cu
  const int64_t red0 = O.bpos ? (int64_t)O.bpos[i] * O.q : O.red_off[i];
  for (int c0 = 0; c0 < V.w; c0 += kChunk) {
    const int cw = min(kChunk, V.w - c0);
    T C[kMaxRows * kChunk];
    for (int c = 0; c < cw; ++c) {
      for (int r = 0; r < n; ++r) C[c * na + r] = V.S[V.row_off[i] * V.w + (int64_t)(c0 + c) * n + r];
      for (int r = n; r < na; ++r) C[c * na + r] = 0;
    }
    for (int k = 0; k < m; ++k) {
      const T* x = B + k * na;
      for (int c = 0; c < cw; ++c) {
        T* y = C + c * na;
        T w = y[k];
        for (int r = k + 1; r < na; ++r) w += x[r] * y[r];
        w *= tau[k];
        y[k] -= w;
        for (int r = k + 1; r < na; ++r) y[r] -= w * x[r];
      }
    }
    for (int c = 0; c < cw; ++c) {
      for (int r = 0; r < m; ++r) O.R12[(V.col_off[i] + r) * (int64_t)V.w + c0 + c] = C[c * na + r];
      for (int r = m; r < na; ++r) {
        const int64_t row = red0 + (r - m);
        O.Xw[row * V.w + c0 + c] = C[c * na + r];
        if (c0 + c == 0 && O.Xstart) O.Xstart[row] = V.start[i];
      }
    }
  }
}

// Damping rows of the shared columns (dense case), s rows from row0, and with `damp` false zero rows
// that pad the first level: `count` rows in all.
template <typename T>
__global__ void reduced_damping_kernel(T* X0, int64_t ld0, int64_t row0, int s, int count, bool damp, const double* D,
                                       int64_t nb, double lam_half) {
  dev::chain_wait();
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)count * s) return;
  const int c = (int)(e / count), j = (int)(e % count);
  X0[(int64_t)c * ld0 + row0 + j] = (damp && c == j) ? (T)(lam_half * D[nb + j]) : T(0);
}

// Per-block Q_i^T [b_i; 0]: top m -> ctop, bottom -> reduced rhs rows.  NA > 0: every block has
// at most NA augmented rows and MM columns (loops unrolled to those bounds, registers only).
template <typename T, int NA = 0, int MM = 0>
__global__ void block_apply_qt_kernel(ComposedView<T> V, FactorOut<T> O, const T* b, T* rhs0) {
  dev::chain_wait();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= V.K) return;
  if constexpr (NA > 0) {
    const int n = V.n[i], m = V.m[i];
    const int na = n + (O.damp ? m : 0);
    T y[NA];
#pragma unroll
    for (int r = 0; r < NA; ++r) y[r] = r < n ? b[V.row_off[i] + r] : T(0);
    const T* F = O.Fa + O.aug_off[i];
    const int64_t red0 = O.bpos ? (int64_t)O.bpos[i] * O.q : O.red_off[i];
#pragma unroll
    for (int k = 0; k < MM; ++k) {
      if (k < m) {
        T w = y[k];
#pragma unroll
        for (int r = 0; r < NA; ++r)
          if (r > k && r < na) w += F[k * na + r] * y[r];
        w *= O.tau[V.col_off[i] + k];
        y[k] -= w;
#pragma unroll
        for (int r = 0; r < NA; ++r)
          if (r > k && r < na) y[r] -= w * F[k * na + r];
      }
    }
#pragma unroll
    for (int r = 0; r < NA; ++r) {
      if (r < m) O.ctop[V.col_off[i] + r] = y[r];
      else if (rhs0 && r < na) rhs0[red0 + (r - m)] = y[r];
    }
    return;
  }
  const int n = V.n[i], m = V.m[i];
  const int na = n + (O.damp ? m : 0);
  T y[kMaxRows];
  for (int r = 0; r < n; ++r) y[r] = b[V.row_off[i] + r];
  for (int r = n; r < na; ++r) y[r] = 0;
  const T* F = O.Fa + O.aug_off[i];
  for (int k = 0; k < m; ++k) {
    const T* x = F + k * na;
    T w = y[k];
    for (int r = k + 1; r < na; ++r) w += x[r] * y[r];
    w *= O.tau[V.col_off[i] + k];
    y[k] -= w;
    for (int r = k + 1; r < na; ++r) y[r] -= w * x[r];
  }
  for (int r = 0; r < m; ++r) O.ctop[V.col_off[i] + r] = y[r];
  const int64_t red0 = O.bpos ? (int64_t)O.bpos[i] * O.q : O.red_off[i];
  if (rhs0)
    for (int r = m; r < na; ++r) rhs0[red0 + (r - m)] = y[r];
}

// Per-block R_i x_i = rhs_i - R12_i x_S; rhs from ctop (T) or from a double vector.  NA > 0:
// every block has at most NA augmented rows and MM columns (registers only).
template <typename T, int NA = 0, int MM = 0>
__global__ void block_backsub_kernel(ComposedView<T> V, FactorOut<T> O, const T* rhs_t,
                                     const T* xS, T* x, int accumulate) {
  dev::chain_wait();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= V.K) return;
  if constexpr (NA > 0) {
    const int n = V.n[i], m = V.m[i];
    const int na = n + (O.damp ? m : 0);
    const int64_t c0 = V.col_off[i];
    const int64_t st = V.coupled == QRKIT_COUPLED_WINDOW ? V.start[i] : 0;
    T y[MM];
#pragma unroll
    for (int k = 0; k < MM; ++k) {
      T v = T(0);
      if (k < m) {
        v = rhs_t[c0 + k];
        if (V.coupled != QRKIT_COUPLED_NONE && xS) {
          const T* r12 = O.R12 + (c0 + k) * (int64_t)V.w;
          for (int t = 0; t < V.w; ++t)
            if (st + t < V.s) v -= r12[t] * xS[st + t];
        }
      }
      y[k] = v;
    }
    const T* F = O.Fa + O.aug_off[i];
#pragma unroll
    for (int k = MM - 1; k >= 0; --k) {
      if (k < m) {
        T v = y[k];
#pragma unroll
        for (int j = k + 1; j < MM; ++j)
          if (j < m) v -= F[j * na + k] * y[j];
        y[k] = v / F[k * na + k];
      }
    }
#pragma unroll
    for (int k = 0; k < MM; ++k)
      if (k < m) x[c0 + k] = accumulate ? x[c0 + k] + y[k] : y[k];
    return;
  }
  const int n = V.n[i], m = V.m[i];
  const int na = n + (O.damp ? m : 0);
  const int64_t c0 = V.col_off[i];
  T y[kMaxCols];
  for (int k = 0; k < m; ++k) {
    T v = rhs_t[c0 + k];
    if (V.coupled != QRKIT_COUPLED_NONE && xS) {
      const int64_t st = V.coupled == QRKIT_COUPLED_WINDOW ? V.start[i] : 0;
      const T* r12 = O.R12 + (c0 + k) * (int64_t)V.w;
      for (int t = 0; t < V.w; ++t)
        if (st + t < V.s) v -= r12[t] * xS[st + t];
    }
    y[k] = v;
  }
  const T* F = O.Fa + O.aug_off[i];
  for (int k = m - 1; k >= 0; --k) {
    T v = y[k];
    for (int j = k + 1; j < m; ++j) v -= F[j * na + k] * y[j];
    y[k] = v / F[k * na + k];
  }
  for (int k = 0; k < m; ++k) x[c0 + k] = accumulate ? x[c0 + k] + y[k] : y[k];
}

// ---- refinement: g = J^T (b - J p) - lambda D^2 p of double plans, and of float plans without a dense S whose blocks
// differ in shape (a dense S: dense_solve.cu; blocks of one shape with windows: window_sums.cu).  In double; blocks of
// floats up to 6 x 2 sum their rows in float pairs ----
constexpr int kCtaSumCols = 4096;   // dense S: shared columns summed per CTA in shared memory
constexpr int kWinSumCols = 2048;   // windowed S: the column range of a CTA summed in shared memory

template <typename T>
__device__ __forceinline__ void resid_g_block(ComposedView<T> V, const T* b, const T* p, const double* D,
                                              double lam, double* g, double* gS, int64_t goff, int64_t i) {
  const int n = V.n[i], m = V.m[i];
  const int64_t c0 = V.col_off[i], r0 = V.row_off[i];
  const T* J = V.J + V.val_off[i];
  const int64_t st = V.coupled == QRKIT_COUPLED_WINDOW ? V.start[i] : 0;
  const bool dense = sizeof(T) == sizeof(double) && V.coupled == QRKIT_COUPLED_DENSE;   // float: dense_solve.cu
  double res[kMaxRows];
  for (int r = 0; r < n; ++r) {
    double acc = (double)b[r0 + r];
    for (int j = 0; j < m; ++j) acc -= (double)J[j * n + r] * (double)p[c0 + j];
    if (dense) {
      for (int c = 0; c < V.s; ++c)
        acc -= (double)V.S[(int64_t)c * V.rows + r0 + r] * (double)p[V.nb + c];
    } else if (V.coupled == QRKIT_COUPLED_WINDOW) {
      for (int t = 0; t < V.w; ++t)
        if (st + t < V.s) acc -= (double)V.S[r0 * V.w + (int64_t)t * n + r] * (double)p[V.nb + st + t];
    }
    res[r] = acc;
  }
  for (int j = 0; j < m; ++j) {
    double acc = 0;
    for (int r = 0; r < n; ++r) acc += (double)J[j * n + r] * res[r];
    const double d = D[c0 + j];
    g[c0 + j] = acc - lam * d * d * (double)p[c0 + j];
  }
  if (dense) {
    for (int c = 0; c < V.s; ++c) {
      double acc = 0;
      for (int r = 0; r < n; ++r) acc += (double)V.S[(int64_t)c * V.rows + r0 + r] * res[r];
      if (acc != 0.0) atomicAdd(&gS[c], acc);
    }
  } else if (V.coupled == QRKIT_COUPLED_WINDOW) {
    for (int t = 0; t < V.w; ++t) {
      double acc = 0;
      for (int r = 0; r < n; ++r) acc += (double)V.S[r0 * V.w + (int64_t)t * n + r] * res[r];
      if (acc != 0.0 && st + t < V.s) atomicAdd(&gS[st + t - goff], acc);
    }
  }
}

// resid_g_small for float data: the residual b - J p - S p_S and the sums J^T r, S^T r in
// compensated float arithmetic (as if in twice the working precision) instead of FP64, whose
// rate on this part is a small fraction of FP32's; each sum is rounded to double once, for g
// and the column accumulation.
template <int NR, int MM>
__device__ __forceinline__ void resid_g_small_f32(const ComposedView<float>& V, const float* b, const float* p,
                                                  const double* D, double lam, double* g, double* gS, int64_t goff,
                                                  int64_t i) {
  const int n = V.n[i], m = V.m[i];
  const int64_t c0 = V.col_off[i], r0 = V.row_off[i];
  const float* J = V.J + V.val_off[i];
  const int64_t st = V.coupled == QRKIT_COUPLED_WINDOW ? V.start[i] : 0;
  if constexpr (MM == 1 && NR >= 2) {
    // the 2 x 1 point blocks of curve fits with windows of 8: the window (2 x 8 column-major,
    // 32-byte aligned in a 16-byte aligned S) by four 16-byte loads
    if (V.coupled == QRKIT_COUPLED_WINDOW && V.w == 8 && n == 2 && m == 1 &&
        (reinterpret_cast<uintptr_t>(V.S) & 15) == 0) {
      const float4* s4 = reinterpret_cast<const float4*>(V.S + r0 * 8);
      float sv[16];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 v = s4[q];
        sv[4 * q] = v.x;
        sv[4 * q + 1] = v.y;
        sv[4 * q + 2] = v.z;
        sv[4 * q + 3] = v.w;
      }
      const float p0 = p[c0];
      float ps[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) ps[t] = st + t < V.s ? p[V.nb + st + t] : 0.f;
      float rh2[2], rl2[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float sh = b[r0 + r], sl = 0.f;
        dev::dot2(sh, sl, -J[r], p0);
#pragma unroll
        for (int t = 0; t < 8; ++t) dev::dot2(sh, sl, -sv[2 * t + r], ps[t]);
        rh2[r] = sh;
        rl2[r] = sl;
      }
      {
        float ah = 0.f, al = 0.f;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          dev::dot2(ah, al, J[r], rh2[r]);
          al = __fmaf_rn(J[r], rl2[r], al);
        }
        const double d = D[c0];
        g[c0] = ((double)ah + (double)al) - lam * d * d * (double)p0;
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        float ah = 0.f, al = 0.f;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          dev::dot2(ah, al, sv[2 * t + r], rh2[r]);
          al = __fmaf_rn(sv[2 * t + r], rl2[r], al);
        }
        const double acc = (double)ah + (double)al;
        if (acc != 0.0 && st + t < V.s) atomicAdd(&gS[st + t - goff], acc);
      }
      return;
    }
  }
  float pj[MM], rh[NR], rl[NR];
#pragma unroll
  for (int j = 0; j < MM; ++j) pj[j] = j < m ? p[c0 + j] : 0.f;
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    float sh = 0.f, sl = 0.f;
    if (r < n) {
      sh = b[r0 + r];
#pragma unroll
      for (int j = 0; j < MM; ++j)
        if (j < m) dev::dot2(sh, sl, -J[j * n + r], pj[j]);
      if (V.coupled == QRKIT_COUPLED_WINDOW) {
        for (int t = 0; t < V.w; ++t)
          if (st + t < V.s) dev::dot2(sh, sl, -V.S[r0 * V.w + (int64_t)t * n + r], p[V.nb + st + t]);
      }
    }
    rh[r] = sh;
    rl[r] = sl;
  }
  // a sum of a x over the rows with x = rh + rl: the rh part compensated, the rl part plain
#pragma unroll
  for (int j = 0; j < MM; ++j) {
    if (j < m) {
      float ah = 0.f, al = 0.f;
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (r < n) {
          const float a = J[j * n + r];
          dev::dot2(ah, al, a, rh[r]);
          al = __fmaf_rn(a, rl[r], al);
        }
      const double d = D[c0 + j];
      g[c0 + j] = ((double)ah + (double)al) - lam * d * d * (double)pj[j];
    }
  }
  if (V.coupled == QRKIT_COUPLED_WINDOW) {
    for (int t = 0; t < V.w; ++t) {
      float ah = 0.f, al = 0.f;
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (r < n) {
          const float a = V.S[r0 * V.w + (int64_t)t * n + r];
          dev::dot2(ah, al, a, rh[r]);
          al = __fmaf_rn(a, rl[r], al);
        }
      const double acc = (double)ah + (double)al;
      if (acc != 0.0 && st + t < V.s) atomicAdd(&gS[st + t - goff], acc);
    }
  }
}

// resid_g_block for blocks of at most NR rows and MM columns, every array in registers.
template <typename T, int NR, int MM>
__device__ __forceinline__ void resid_g_small(const ComposedView<T>& V, const T* b, const T* p, const double* D,
                                              double lam, double* g, double* gS, int64_t goff, int64_t i) {
  if constexpr (sizeof(T) == sizeof(float)) {
    resid_g_small_f32<NR, MM>(V, b, p, D, lam, g, gS, goff, i);
    return;
  }
  const int n = V.n[i], m = V.m[i];
  const int64_t c0 = V.col_off[i], r0 = V.row_off[i];
  const T* J = V.J + V.val_off[i];
  const int64_t st = V.coupled == QRKIT_COUPLED_WINDOW ? V.start[i] : 0;
  double pj[MM], res[NR];
#pragma unroll
  for (int j = 0; j < MM; ++j) pj[j] = j < m ? (double)p[c0 + j] : 0.0;
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    double acc = 0.0;
    if (r < n) {
      acc = (double)b[r0 + r];
#pragma unroll
      for (int j = 0; j < MM; ++j)
        if (j < m) acc -= (double)J[j * n + r] * pj[j];
      if (V.coupled == QRKIT_COUPLED_DENSE) {
        for (int c = 0; c < V.s; ++c) acc -= (double)V.S[(int64_t)c * V.rows + r0 + r] * (double)p[V.nb + c];
      } else if (V.coupled == QRKIT_COUPLED_WINDOW) {
        for (int t = 0; t < V.w; ++t)
          if (st + t < V.s) acc -= (double)V.S[r0 * V.w + (int64_t)t * n + r] * (double)p[V.nb + st + t];
      }
    }
    res[r] = acc;
  }
#pragma unroll
  for (int j = 0; j < MM; ++j) {
    if (j < m) {
      double acc = 0;
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (r < n) acc += (double)J[j * n + r] * res[r];
      const double d = D[c0 + j];
      g[c0 + j] = acc - lam * d * d * pj[j];
    }
  }
  if (V.coupled == QRKIT_COUPLED_DENSE) {
    for (int c = 0; c < V.s; ++c) {
      double acc = 0;
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (r < n) acc += (double)V.S[(int64_t)c * V.rows + r0 + r] * res[r];
      if (acc != 0.0) atomicAdd(&gS[c], acc);
    }
  } else if (V.coupled == QRKIT_COUPLED_WINDOW) {
    for (int t = 0; t < V.w; ++t) {
      double acc = 0;
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (r < n) acc += (double)V.S[r0 * V.w + (int64_t)t * n + r] * res[r];
      if (acc != 0.0 && st + t < V.s) atomicAdd(&gS[st + t - goff], acc);
    }
  }
}

// Windowed S: the columns the CTA's blocks touch, [lo, hi) with hi = max start + w (uniform
// over the CTA; blocks past K do not count).  The kernels sum into shared memory when the range
// fits (consecutive blocks of one LM problem share its few hundred columns), so a column leaves
// the CTA with one global atomic instead of one per block.
template <typename T>
__device__ __forceinline__ bool window_range(const ComposedView<T>& V, int64_t i, int cap, int64_t& lo, int& width) {
  __shared__ unsigned long long rng[2];
  if (threadIdx.x == 0) {
    rng[0] = ~0ull;
    rng[1] = 0ull;
  }
  __syncthreads();
  unsigned long long mn = ~0ull, mx = 0ull;
  if (i < V.K) mn = mx = (unsigned long long)V.start[i];
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, d));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, d));
  }
  if ((threadIdx.x & 31) == 0 && mn != ~0ull) {
    atomicMin(&rng[0], mn);
    atomicMax(&rng[1], mx);
  }
  __syncthreads();
  if (rng[0] == ~0ull) return false;
  lo = (int64_t)rng[0];
  const int64_t w = (int64_t)rng[1] + V.w - lo;
  width = (int)(w < (int64_t)cap ? w : (int64_t)cap);
  return w <= cap;
}

template <typename T, int NA = 0, int MM = 0>
__global__ void resid_g_kernel(ComposedView<T> V, const T* b, const T* p, const double* D,
                               double lam, double* g, double* gS, int win_cols) {
  dev::chain_wait();
  // dense S: every block adds to all s shared columns; the CTA's sums are gathered in shared
  // memory and leave with one global atomic per column
  extern __shared__ double sgS[];
  const bool cta_sum = sizeof(T) == sizeof(double) && V.coupled == QRKIT_COUPLED_DENSE && V.s <= kCtaSumCols;
  if (cta_sum) {
    for (int c = threadIdx.x; c < V.s; c += blockDim.x) sgS[c] = 0.0;
    __syncthreads();
  }
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int64_t lo = 0;
  int width = 0;
  const bool win_sum = V.coupled == QRKIT_COUPLED_WINDOW && win_cols > 0 && window_range(V, i, win_cols, lo, width);
  if (win_sum) {
    for (int c = threadIdx.x; c < width; c += blockDim.x) sgS[c] = 0.0;
    __syncthreads();
  }
  if (i < V.K) {
    if constexpr (NA > 0)
      resid_g_small<T, NA, MM>(V, b, p, D, lam, g, (cta_sum || win_sum) ? sgS : gS, win_sum ? lo : 0, i);
    else
      resid_g_block(V, b, p, D, lam, g, (cta_sum || win_sum) ? sgS : gS, win_sum ? lo : 0, i);
  }
  if (cta_sum) {
    __syncthreads();
    for (int c = threadIdx.x; c < V.s; c += blockDim.x)
      if (sgS[c] != 0.0) atomicAdd(&gS[c], sgS[c]);
  }
  if (win_sum) {
    __syncthreads();
    for (int c = threadIdx.x; c < width; c += blockDim.x)
      if (sgS[c] != 0.0) atomicAdd(&gS[lo + c], sgS[c]);
  }
}

__global__ void gS_damping_kernel(double* gS, const float* pf, const double* pd, const double* D,
                                  int64_t nb, int s, double lam) {
  dev::chain_wait();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= s) return;
  const double pv = pf ? (double)pf[nb + c] : pd[nb + c];
  const double d = D[nb + c];
  gS[c] -= lam * d * d * pv;
}

// h_i = R_i^{-T} g_i per block; then gS -= R12_i^T h_i (dense S: summed per CTA first).
template <typename T>
__device__ __forceinline__ void fwdsub_rt_block(ComposedView<T> V, FactorOut<T> O, const double* g, T* h,
                                                double* gS, int64_t goff, int64_t i) {
  const int n = V.n[i], m = V.m[i];
  const int na = n + (O.damp ? m : 0);
  const int64_t c0 = V.col_off[i];
  const T* F = O.Fa + O.aug_off[i];
  T hv[kMaxCols];
  for (int k = 0; k < m; ++k) {
    T v = (T)g[c0 + k];
    for (int j = 0; j < k; ++j) v -= F[k * na + j] * hv[j];
    hv[k] = v / F[k * na + k];
    h[c0 + k] = hv[k];
  }
  if (V.coupled != QRKIT_COUPLED_NONE) {
    const int64_t st = V.coupled == QRKIT_COUPLED_WINDOW ? V.start[i] : 0;
    for (int t = 0; t < V.w; ++t) {
      if (st + t >= V.s) continue;
      double acc = 0;
      for (int k = 0; k < m; ++k) acc += (double)O.R12[(c0 + k) * (int64_t)V.w + t] * (double)hv[k];
      if (acc != 0.0) atomicAdd(&gS[st + t - goff], -acc);
    }
  }
}

// fwdsub_rt_block for blocks of at most NA augmented rows and MM columns (registers only).
template <typename T, int NA, int MM>
__device__ __forceinline__ void fwdsub_rt_small(const ComposedView<T>& V, const FactorOut<T>& O, const double* g, T* h,
                                                double* gS, int64_t goff, int64_t i) {
  const int n = V.n[i], m = V.m[i];
  const int na = n + (O.damp ? m : 0);
  const int64_t c0 = V.col_off[i];
  const T* F = O.Fa + O.aug_off[i];
  T hv[MM];
#pragma unroll
  for (int k = 0; k < MM; ++k) {
    T v = T(0);
    if (k < m) {
      v = (T)g[c0 + k];
#pragma unroll
      for (int j = 0; j < MM; ++j)
        if (j < k) v -= F[k * na + j] * hv[j];
      v = v / F[k * na + k];
      h[c0 + k] = v;
    }
    hv[k] = v;
  }
  if (V.coupled != QRKIT_COUPLED_NONE) {
    const int64_t st = V.coupled == QRKIT_COUPLED_WINDOW ? V.start[i] : 0;
    if constexpr (sizeof(T) == 4 && MM == 1) {
      if (V.coupled == QRKIT_COUPLED_WINDOW && V.w == 8 && m == 1) {
        // one column: R12 row by two 16-byte loads (32-byte aligned), the products in float
        // (h is itself a float correction), each rounded to double once for the sum
        const float4* r4 = reinterpret_cast<const float4*>(O.R12 + c0 * 8);
        const float4 a = r4[0], bq = r4[1];
        const float rv[8] = {a.x, a.y, a.z, a.w, bq.x, bq.y, bq.z, bq.w};
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const float prod = rv[t] * hv[0];
          if (prod != 0.f && st + t < V.s) atomicAdd(&gS[st + t - goff], -(double)prod);
        }
        return;
      }
    }
    for (int t = 0; t < V.w; ++t) {
      if (st + t >= V.s) continue;
      double acc = 0;
#pragma unroll
      for (int k = 0; k < MM; ++k)
        if (k < m) acc += (double)O.R12[(c0 + k) * (int64_t)V.w + t] * (double)hv[k];
      if (acc != 0.0) atomicAdd(&gS[st + t - goff], -acc);
    }
  }
}

template <typename T, int NA = 0, int MM = 0>
__global__ void block_fwdsub_rt_kernel(ComposedView<T> V, FactorOut<T> O, const double* g, T* h,
                                       double* gS, int win_cols) {
  dev::chain_wait();
  extern __shared__ double sgS[];
  const bool cta_sum = sizeof(T) == sizeof(double) && V.coupled == QRKIT_COUPLED_DENSE && V.s <= kCtaSumCols;
  if (cta_sum) {
    for (int c = threadIdx.x; c < V.s; c += blockDim.x) sgS[c] = 0.0;
    __syncthreads();
  }
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int64_t lo = 0;
  int width = 0;
  const bool win_sum = V.coupled == QRKIT_COUPLED_WINDOW && win_cols > 0 && window_range(V, i, win_cols, lo, width);
  if (win_sum) {
    for (int c = threadIdx.x; c < width; c += blockDim.x) sgS[c] = 0.0;
    __syncthreads();
  }
  if (i < V.K) {
    if constexpr (NA > 0)
      fwdsub_rt_small<T, NA, MM>(V, O, g, h, (cta_sum || win_sum) ? sgS : gS, win_sum ? lo : 0, i);
    else
      fwdsub_rt_block(V, O, g, h, (cta_sum || win_sum) ? sgS : gS, win_sum ? lo : 0, i);
  }
  if (cta_sum) {
    __syncthreads();
    for (int c = threadIdx.x; c < V.s; c += blockDim.x)
      if (sgS[c] != 0.0) atomicAdd(&gS[c], sgS[c]);
  }
  if (win_sum) {
    __syncthreads();
    for (int c = threadIdx.x; c < width; c += blockDim.x)
      if (sgS[c] != 0.0) atomicAdd(&gS[lo + c], sgS[c]);
  }
}

template <typename T>
__global__ void gS_to_T_kernel(const double* gS, T* out, int s) {
  dev::chain_wait();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < s) out[c] = (T)gS[c];
}

template <typename T>
__global__ void axpy_kernel(T* x, const T* d, int64_t n) {
  dev::chain_wait();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) x[i] += d[i];
}

__global__ void widen_kernel(const float* in, double* out, int64_t n) {
  dev::chain_wait();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) out[i] = (double)in[i];
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// ---------------------------------------------------------------------------------------
// Host orchestration.

template <typename T>
static ComposedView<T> view(qrkit_ctx* ctx, const void* J, const void* S) {
  Plan& P = ctx->plan;
  ComposedView<T> V;
  V.K = P.K;
  V.n = (const uint8_t*)P.d_n.ptr;
  V.m = (const uint8_t*)P.d_m.ptr;
  V.val_off = (const int64_t*)P.d_val_off.ptr;
  V.row_off = (const int64_t*)P.d_row_off.ptr;
  V.col_off = (const int64_t*)P.d_col_off.ptr;
  V.start = (const int32_t*)P.d_start.ptr;
  V.coupled = P.s.coupled_kind;
  V.s = (int)P.s.shared_cols;
  V.w = P.s.coupled_kind == QRKIT_COUPLED_DENSE ? (int)P.s.shared_cols : P.s.window;
  V.rows = P.rows;
  V.nb = P.cols;
  V.J = (const T*)J;
  V.S = (const T*)S;
  return V;
}

// Rows of the dense reduced block before the stacked bottoms.  With column panels the damping rows of
// the shared columns come first: row c of a tile moves up by 32 with every panel, so each of them is
// the pivot row of its own column, and a column that is zero but for it stays exactly zero elsewhere.
static int64_t reduced_head(const qrkit_ctx* ctx) {
  const Composed& C = ctx->comp;
  return C.damp && !C.panels.empty() ? ctx->plan.s.shared_cols : 0;
}

template <typename T>
static FactorOut<T> fout(qrkit_ctx* ctx) {
  Composed& C = ctx->comp;
  FactorOut<T> O;
  O.damp = C.damp;
  O.lam_half = C.lam_half;
  O.D = (const double*)C.D.ptr;
  O.Fa = (T*)C.Fa.ptr;
  O.tau = (T*)C.tau.ptr;
  O.R12 = (T*)C.R12.ptr;
  O.ctop = (T*)C.ctop.ptr;
  O.aug_off = (const int64_t*)(C.damp ? C.d_aug_off_d.ptr : C.d_aug_off_u.ptr);
  O.red_off = (const int64_t*)(C.damp ? C.d_red_off_d.ptr : C.d_red_off_u.ptr);
  O.X0 = C.levels.empty() ? nullptr : (T*)C.levels[0].X.ptr + reduced_head(ctx);
  O.ld0 = C.levels.empty() ? 0 : C.levels[0].ld;
  O.Xw = (T*)(C.bins ? C.Xw_s.ptr : C.Xw.ptr);
  O.Xstart = C.bins ? nullptr : (int64_t*)C.Xstart.ptr;
  O.bpos = C.bins ? (const int32_t*)C.bpos.ptr : nullptr;
  O.q = C.bins ? (int)(C.red_rows / ctx->plan.K) : 0;
  O.status = ctx->d_status;
  return O;
}

#define LAUNCH(ctx, ...)                                  \
  do {                                                    \
    __VA_ARGS__;                                          \
    (ctx)->launches += 1;                                 \
    QRKIT_CUDA_TRY(ctx, cudaGetLastError());              \
  } while (0)

// Shape class of a plan's blocks for the per-block kernels: 1 if every augmented block is at
// most 3 x 1, 2 if at most 6 x 2, else 0 (the general kernels with runtime loops).
int small_class(const Plan& P, bool damp) {
  const int na = P.max_n + (damp ? P.max_m : 0);
  if (P.max_m == 1 && na <= 3) return 1;
  if (P.max_m <= 2 && na <= 6) return 2;
  return 0;
}
// A per-block kernel template KERNEL<T, NA, MM> launched in the instantiation of the class.
#define LAUNCH_SHAPED(ctx, chained, cls, KERNEL, grid, threads, smem, stream, ...)                                     \
  do {                                                                                                                \
    if ((cls) == 1) LAUNCH(ctx, (launch_kernel(chained, stream, grid, threads, smem, (KERNEL<T, 3, 1>), __VA_ARGS__))); \
    else if ((cls) == 2)                                                                                              \
      LAUNCH(ctx, (launch_kernel(chained, stream, grid, threads, smem, (KERNEL<T, 6, 2>), __VA_ARGS__)));              \
    else LAUNCH(ctx, (launch_kernel(chained, stream, grid, threads, smem, KERNEL<T>, __VA_ARGS__)));                   \
  } while (0)

// R_i x_i = rhs_i - R12_i x_S for every block.  From 16 shared columns on in dense_solve.cu; below, and for windows of
// up to 8, a thread per block.
template <typename T>
static qrkit_status launch_block_backsub(qrkit_ctx* ctx, bool chained, const ComposedView<T>& V, const FactorOut<T>& O,
                                         const T* rhs, const T* xS, T* x, int accumulate) {
  if (V.coupled == QRKIT_COUPLED_DENSE && V.s >= 16)
    return dense_block_backsub<T>(ctx, chained, V, O, rhs, xS, x, accumulate);
  if (window21(ctx)) return window21_backsub<T>(ctx, V, O, rhs, xS, x, accumulate);
  LAUNCH_SHAPED(ctx, chained, small_class(ctx->plan, O.damp), block_backsub_kernel, blocks_for(V.K, 64), 64, 0,
                ctx->stream, V, O, rhs, xS, x, accumulate);
  return QRKIT_OK;
}

template <typename T>
static WindowSums<T> window_sums(qrkit_ctx* ctx, const ComposedView<T>& V, double* out) {
  const Composed& C = ctx->comp;
  WindowSums<T> A{};
  A.K = V.K;
  A.n = ctx->plan.max_n;
  A.m = ctx->plan.max_m;
  A.w = V.w;
  A.s = V.s;
  A.bord = (const int32_t*)C.bord.ptr;
  A.start = V.start;
  A.S = V.S;
  A.R12 = (const T*)C.R12.ptr;
  A.r = (const T*)C.wres.ptr;
  A.h = (const T*)C.h.ptr;
  A.out = out;
  return A;
}

// D = column norms of J (Sec. 5.2), zero -> 1, in double; C.sq is the scratch.  sorted: the plan's blocks have
// been sorted by their window starts.
template <typename T>
static qrkit_status norms_typed(qrkit_ctx* ctx, const ComposedView<T>& V, double* D, bool sorted) {
  Plan& P = ctx->plan;
  Composed& C = ctx->comp;
  cudaStream_t st = ctx->stream;
  const int64_t N = P.cols + P.s.shared_cols;
  qrkit_status rc;
  // dense S: the chunk sums of pass 1 follow the N column sums in the same scratch
  const int64_t nchunk = V.coupled == QRKIT_COUPLED_DENSE ? std::max<int64_t>(1, (V.rows + kNormRows - 1) / kNormRows) : 0;
  const size_t sq_bytes = (size_t)(N + nchunk * (V.coupled == QRKIT_COUPLED_DENSE ? V.s : 0)) * sizeof(double);
  if ((rc = ensure(ctx, C.sq, sq_bytes, "column sums")) != QRKIT_OK) return rc;
  double* sq = (double*)C.sq.ptr;
  QRKIT_CUDA_TRY(ctx, cudaMemsetAsync(sq, 0, (size_t)N * sizeof(double), st));
  LAUNCH(ctx, chain_launch(st, blocks_for(P.K, 128), 128, 0, colnorm_blocks_kernel<T>, V, sq));
  if (V.coupled == QRKIT_COUPLED_DENSE) {
    if (nchunk > (int64_t)INT32_MAX) return fail(ctx, QRKIT_EUNSUPPORTED, "too many rows for the column norms");
    const dim3 grid((unsigned)nchunk, (unsigned)std::min<int64_t>(V.s, 65535));
    LAUNCH(ctx, chain_launch(st, grid, kNormThreads, 0, colnorm_dense_part_kernel<T>, V, sq + N, nchunk));
    LAUNCH(ctx, chain_launch(st, blocks_for(V.s, 128), 128, 0, colnorm_dense_sum_kernel, sq + N, nchunk, V.s,
                             sq + V.nb));
  } else if (V.coupled == QRKIT_COUPLED_WINDOW && sorted) {
    const WindowSums<T> A = window_sums<T>(ctx, V, sq + V.nb);
    if ((rc = window_square_sums<T>(ctx, A)) != QRKIT_OK) return rc;
  } else if (V.coupled == QRKIT_COUPLED_WINDOW) {
    LAUNCH(ctx, chain_launch(st, blocks_for(P.K, 128), 128, 0, colnorm_window_kernel<T>, V, sq));
  }
  LAUNCH(ctx, chain_launch(st, blocks_for(N, 256), 256, 0, finalize_norms_kernel, sq, D, N));
  return QRKIT_OK;
}

// Column-panel TSQR of a float dense reduced block (s a multiple of 32 above 32).  Panel j
// (columns c0 = 32 j ..): its levels are factored tile by tile (R rows up; the top level's into
// R_S), and after each level the tiles' Q^T is applied to the panel's trailing columns on the
// tensor cores, whose rows move up with the R rows or down into the next panel's first level.
// Narrow panels keep the column-by-column part of the work (the tile QR) small: it grows with the
// panel width, while the trailing updates do the rest of the arithmetic.
static qrkit_status factor_panels(qrkit_ctx* ctx, int s) {
  Composed& C = ctx->comp;
  float* Rs = (float*)C.Rs.ptr;
  const int np = 1 + (int)C.panels.size();
  for (int j = 0; j < np; ++j) {
    std::vector<TsqrLevel>& LV = j == 0 ? C.levels : C.panels[j - 1].levels;
    const int c0 = j * kPanelCols;
    const int n = s - c0 - kPanelCols;   // trailing columns
    for (size_t l = 0; l < LV.size(); ++l) {
      TsqrLevel& L = LV[l];
      const bool top = l + 1 == LV.size();
      float* X = (float*)L.X.ptr;
      const int64_t ldn = top ? s : LV[l + 1].ld;
      float* Xn = top ? Rs + (int64_t)c0 * s + c0 : (float*)LV[l + 1].X.ptr;
      qrkit_status rc = tsqr_panel_tile(ctx, X, L.ld, L.M, Xn, ldn, L.tiles, (float*)L.T.ptr,
                                        (float*)L.tau.ptr);
      if (rc != QRKIT_OK) return rc;
      if (n > 0) {
        TsqrLevel& N0 = C.panels[j].levels[0];
        rc = tsqr_panel_apply(ctx, X, L.ld, L.M, (const float*)L.T.ptr, n, Xn + kPanelCols * ldn, ldn,
                              (float*)N0.X.ptr, N0.ld, L.down0, L.tiles);
        if (rc != QRKIT_OK) return rc;
      }
    }
  }
  return QRKIT_OK;
}

template <typename T>
static qrkit_status factor_typed(qrkit_ctx* ctx, const void* J, const void* S, const void* Dext,
                                 double lambda, bool dext_double = false, bool sorted = false) {
  Plan& P = ctx->plan;
  Composed& C = ctx->comp;
  cudaStream_t st = ctx->stream;
  const int64_t N = P.cols + P.s.shared_cols;
  qrkit_status rc;
  if ((rc = ensure(ctx, C.D, (size_t)N * sizeof(double), "D")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.sq, (size_t)N * sizeof(double), "column sums")) != QRKIT_OK) return rc;
  C.damp = lambda > 0.0;
  C.lam = lambda;
  C.lam_half = sqrt(lambda);
  if ((rc = composed_layout(ctx, sizeof(T))) != QRKIT_OK) return rc;
  ComposedView<T> V = view<T>(ctx, J, S);
  if (!sorted && (rc = composed_sort_blocks(ctx, &sorted)) != QRKIT_OK) return rc;
  // D: caller's (copied to double) or column norms of J
  if (Dext) {
    if (sizeof(T) == sizeof(double) || dext_double) {
      QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(C.D.ptr, Dext, (size_t)N * sizeof(double),
                                          cudaMemcpyDeviceToDevice, st));
    } else {
      rc = widen_to_double(ctx, (const float*)Dext, (double*)C.D.ptr, N);
      if (rc != QRKIT_OK) return rc;
    }
  } else if ((rc = norms_typed<T>(ctx, V, (double*)C.D.ptr, sorted)) != QRKIT_OK) {
    return rc;
  }
  FactorOut<T> O = fout<T>(ctx);
  // the small-block kernels when every block fits them (e.g. 2 x 1 blocks of curve fits)
  const int cls = small_class(P, O.damp);
  if (window21(ctx) && (reinterpret_cast<uintptr_t>(V.S) & 15) == 0) {
    if ((rc = window21_factor<T>(ctx, V, O)) != QRKIT_OK) return rc;
  } else if (cls == 1)
    LAUNCH(ctx, (chain_launch(st, blocks_for(P.K, 128), 128, 0, (block_factor_small_kernel<T, 3, 1>), V, O)));
  else if (cls == 2)
    LAUNCH(ctx, (chain_launch(st, blocks_for(P.K, 128), 128, 0, (block_factor_small_kernel<T, 6, 2>), V, O)));
  else
    LAUNCH(ctx, chain_launch(st, blocks_for(P.K, 64), 64, 0, block_factor_kernel<T>, V, O));
  if (V.coupled == QRKIT_COUPLED_DENSE && (rc = dense_apply_blocks<T>(ctx, V, O)) != QRKIT_OK) return rc;
  if (V.coupled == QRKIT_COUPLED_WINDOW && !C.bins) {
    // P_r of the reduced block: its rows sorted by leading column per segment (Sec. 4.3)
    rc = reduced_row_sort(ctx, C.sort, (int64_t)P.seg_cols.size(), C.sort_hist_entries,
                          (const int64_t*)C.Xstart.ptr, C.Xw.ptr, V.w, (int*)C.hist.ptr,
                          (int64_t*)C.spos.ptr, (int64_t*)C.order.ptr, (int64_t*)C.Xstart_s.ptr, C.Xw_s.ptr);
    if (rc != QRKIT_OK) return rc;
  }
  if (V.coupled == QRKIT_COUPLED_DENSE) {
    const int s = V.s;
    T* X0 = (T*)C.levels[0].X.ptr;
    if (C.damp)
      LAUNCH(ctx, chain_launch(st, blocks_for((int64_t)s * s, 256), 256, 0, reduced_damping_kernel<T>, X0,
                               C.levels[0].ld, C.panels.empty() ? C.red_rows : 0, s, s, true, (const double*)C.D.ptr,
                               P.cols, C.lam_half));
    const int64_t used = C.red_rows + (C.damp ? s : 0);
    if (C.levels[0].M > used)
      LAUNCH(ctx, chain_launch(st, blocks_for((C.levels[0].M - used) * s, 256), 256, 0, reduced_damping_kernel<T>, X0,
                               C.levels[0].ld, used, s, (int)(C.levels[0].M - used), false, nullptr, 0, 0.0));
    if (!C.panels.empty()) return factor_panels(ctx, s);
    for (size_t l = 0; l < C.levels.size(); ++l) {
      TsqrLevel& L = C.levels[l];
      T* Xn = l + 1 < C.levels.size() ? (T*)C.levels[l + 1].X.ptr : nullptr;
      const int64_t ldn = l + 1 < C.levels.size() ? C.levels[l + 1].ld : 0;
      if ((rc = tsqr_tile<T>(ctx, (T*)L.X.ptr, L.ld, L.M, s, C.tile_rows, (T*)L.tau.ptr, Xn, ldn, L.tiles)) != QRKIT_OK)
        return rc;
    }
  }
  return QRKIT_OK;
}

template <typename T>
static qrkit_status solve_typed(qrkit_ctx* ctx, bool chained, const void* J, const void* S, const void* b, void* p,
                                int refine_steps, bool qt_only, void* qtb_out) {
  Plan& P = ctx->plan;
  Composed& C = ctx->comp;
  cudaStream_t st = ctx->stream;
  ComposedView<T> V = view<T>(ctx, J, S);
  FactorOut<T> O = fout<T>(ctx);
  const int s = V.s;
  const int64_t nb = P.cols;
  T* x = (T*)p;
  // Q^T [b; 0]
  T* rhs0 = (V.coupled == QRKIT_COUPLED_DENSE) ? (T*)C.levels[0].rhs.ptr + reduced_head(ctx)
             : (V.coupled == QRKIT_COUPLED_WINDOW ? (T*)(C.bins ? C.rhs_s.ptr : C.rhs_red.ptr) : nullptr);
  if (window21(ctx)) {
    const qrkit_status rc = window21_qt<T>(ctx, chained, V, O, (const T*)b, rhs0);
    if (rc != QRKIT_OK) return rc;
  } else {
    LAUNCH_SHAPED(ctx, chained, small_class(P, O.damp), block_apply_qt_kernel, blocks_for(P.K, 64), 64, 0, st, V, O,
                  (const T*)b, rhs0);
  }
  if (V.coupled == QRKIT_COUPLED_DENSE) {
    const int64_t head = reduced_head(ctx), tail = C.levels[0].M - head - C.red_rows;   // damping rows and padding
    if (head > 0) QRKIT_CUDA_TRY(ctx, cudaMemsetAsync(C.levels[0].rhs.ptr, 0, (size_t)head * sizeof(T), st));
    if (tail > 0) QRKIT_CUDA_TRY(ctx, cudaMemsetAsync(rhs0 + C.red_rows, 0, (size_t)tail * sizeof(T), st));
    bool done = false;
    if constexpr (sizeof(T) == sizeof(float)) {
      // Q^T of every panel's levels: a level's top rows go up (the last level's into c_S), the
      // others into the next panel's first level
      const int np = 1 + (int)C.panels.size();
      for (int j = 0; j < np && np > 1; ++j) {
        std::vector<TsqrLevel>& LV = j == 0 ? C.levels : C.panels[j - 1].levels;
        float* down = j + 1 < np ? (float*)C.panels[j].levels[0].rhs.ptr : nullptr;
        for (size_t l = 0; l < LV.size(); ++l) {
          TsqrLevel& L = LV[l];
          float* rn = l + 1 < LV.size() ? (float*)LV[l + 1].rhs.ptr : (float*)C.cs.ptr + j * kPanelCols;
          qrkit_status rc = tsqr_panel_qt(ctx, (const float*)L.X.ptr, L.ld, L.M, (const float*)L.tau.ptr,
                                          (const float*)L.rhs.ptr, rn, down, L.down0, L.tiles);
          if (rc != QRKIT_OK) return rc;
        }
        done = true;
      }
    }
    for (size_t l = 0; l < C.levels.size() && !done; ++l) {
      TsqrLevel& L = C.levels[l];
      T* rn = l + 1 < C.levels.size() ? (T*)C.levels[l + 1].rhs.ptr : nullptr;
      qrkit_status rc = tsqr_qt<T>(ctx, (const T*)L.X.ptr, L.ld, L.M, s, C.tile_rows, (const T*)L.tau.ptr,
                                   (T*)L.rhs.ptr, rn, L.tiles);
      if (rc != QRKIT_OK) return rc;
    }
  }
  if (V.coupled == QRKIT_COUPLED_WINDOW && qt_only)
    return fail(ctx, QRKIT_EUNSUPPORTED, "Q^T b is not kept for windowed structures (use qrkit_solve)");
  if (qt_only) {
    // Q^T b reported as [c_blocks (sum m_i); c_S (s)]
    T* out = (T*)qtb_out;
    QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(out, O.ctop, (size_t)nb * sizeof(T), cudaMemcpyDeviceToDevice, st));
    if (s > 0)
      QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(out + nb, C.panels.empty() ? C.levels.back().rhs.ptr : C.cs.ptr,
                                          (size_t)s * sizeof(T), cudaMemcpyDeviceToDevice, st));
    return QRKIT_OK;
  }
  // R_S and c_S: the top level's rows, or the panels' R rows gathered in Rs and cs
  const TsqrLevel* top = C.levels.empty() ? nullptr : &C.levels.back();
  const bool pan = !C.panels.empty();
  const T* RS = pan ? (const T*)C.Rs.ptr : (top ? (const T*)top->X.ptr : nullptr);
  const int64_t ldRS = pan ? s : (top ? top->ld : 0);
  if (V.coupled == QRKIT_COUPLED_DENSE) {
    qrkit_status rc = dense_backsub<T>(ctx, true, RS, ldRS, s, pan ? (const T*)C.cs.ptr : (const T*)top->rhs.ptr, x + nb);
    if (rc != QRKIT_OK) return rc;
  } else if (V.coupled == QRKIT_COUPLED_WINDOW) {
    // reduced banded block of every segment (Sec. 4.4), rows in P_r order, the shared
    // columns' damping rows interleaved
    qrkit_status rc = QRKIT_OK;
    if (!C.bins) rc = reduced_rhs_sort(ctx, (const int64_t*)C.spos.ptr, C.rhs_red.ptr, C.rhs_s.ptr, C.red_rows);
    if (rc != QRKIT_OK) return rc;
    if (C.cr)
      rc = cr_solve(ctx, *C.cr, C.bins ? nullptr : (const int64_t*)C.Xstart_s.ptr,
                    C.bins ? (const int32_t*)C.colptr.ptr : nullptr, C.bins ? O.q : 1, V.w, C.Xw_s.ptr, C.rhs_s.ptr, O.D + nb,
                    C.damp ? C.lam : 0.0, x + nb, (double*)C.res2.ptr);
    else
      rc = banded_explicit_solve(ctx, (int64_t)P.seg_cols.size(), (const int64_t*)C.seg_inst.ptr, C.Xw_s.ptr,
                                 (const int64_t*)C.Xstart_s.ptr, C.rhs_s.ptr, V.w, O.D + nb,
                                 C.damp ? C.lam : 0.0, C.RwS.ptr, C.cS.ptr, x + nb, (double*)C.res2.ptr);
    if (rc != QRKIT_OK) return rc;
  }
  qrkit_status rc_b = launch_block_backsub<T>(ctx, true, V, O, (const T*)O.ctop, s ? x + nb : nullptr, x, 0);
  if (rc_b != QRKIT_OK) return rc_b;
  // refinement (extended-precision residual, corrections through R only)
  for (int it = 0; it < refine_steps; ++it) {
    const int64_t N = nb + s;
    qrkit_status rc;
    if ((rc = ensure(ctx, C.g, (size_t)N * sizeof(double), "refinement g")) != QRKIT_OK) return rc;
    if ((rc = ensure(ctx, C.h, (size_t)N * sizeof(T), "refinement h")) != QRKIT_OK) return rc;
    double* g = (double*)C.g.ptr;
    T* h = (T*)C.h.ptr;
    double* gS = g + nb;
    bool have_g = false;
    if constexpr (sizeof(T) == sizeof(float)) {
      if (V.coupled == QRKIT_COUPLED_DENSE) {   // g_S - R12^T h_B and h_B by row, block and column passes
        if ((rc = dense_refine_gradient(ctx, V, O, (const float*)b, x, C.lam, C.dref.ptr, h, gS)) != QRKIT_OK) return rc;
        have_g = true;
      }
    }
    if (C.bins) {
      QRKIT_CUDA_TRY(ctx, cudaMemsetAsync(gS, 0, (size_t)s * sizeof(double), st));
      WindowSums<T> A = window_sums<T>(ctx, V, gS);
      if ((rc = window_refine_gradient<T>(ctx, V, O, (const T*)b, x, C.lam, A)) != QRKIT_OK) return rc;
      LAUNCH(ctx, chain_launch(st, blocks_for(s, 128), 128, 0, gS_damping_kernel, gS,
                               sizeof(T) == 4 ? (const float*)x : nullptr,
                               sizeof(T) == 8 ? (const double*)x : nullptr, O.D, nb, s, C.lam));
      have_g = true;
    }
    if (!have_g) {
      if (s > 0) QRKIT_CUDA_TRY(ctx, cudaMemsetAsync(gS, 0, (size_t)s * sizeof(double), st));
      // dense S: all s columns per CTA; windowed S: the CTA's column range (up to kWinSumCols),
      // with larger CTAs so that more blocks share a column sum
      const bool win = V.coupled == QRKIT_COUPLED_WINDOW;
      const int rthreads = win ? 256 : 64;
      const size_t sum_smem = (V.coupled == QRKIT_COUPLED_DENSE && s <= kCtaSumCols) ? (size_t)s * sizeof(double)
                              : win ? (size_t)kWinSumCols * sizeof(double) : 0;
      const int win_cols = win ? kWinSumCols : 0;
      LAUNCH_SHAPED(ctx, true, small_class(P, O.damp), resid_g_kernel, blocks_for(P.K, rthreads), rthreads, sum_smem, st, V,
                    (const T*)b, x, O.D, C.lam, g, gS, win_cols);
      if (s > 0)
        LAUNCH(ctx, chain_launch(st, blocks_for(s, 128), 128, 0, gS_damping_kernel, gS,
                                 sizeof(T) == 4 ? (const float*)x : nullptr,
                                 sizeof(T) == 8 ? (const double*)x : nullptr, O.D, nb, s, C.lam));
      LAUNCH_SHAPED(ctx, true, small_class(P, O.damp), block_fwdsub_rt_kernel, blocks_for(P.K, rthreads), rthreads,
                    sum_smem, st, V, O, g, h, gS, win_cols);
    }
    if (V.coupled == QRKIT_COUPLED_WINDOW && C.cr) {
      // dp_S = R_S^{-1} R_S^{-T} (g_S - R12^T h_B) with the parallel banded factor
      if ((rc = cr_normal_solve(ctx, *C.cr, gS, h + nb, x + nb)) != QRKIT_OK) return rc;
    } else if (V.coupled == QRKIT_COUPLED_WINDOW) {
      // h_S = R_S^{-T} (g_S - R12^T h_B), then dp_S = R_S^{-1} h_S, both banded
      LAUNCH(ctx, chain_launch(st, blocks_for(s, 128), 128, 0, gS_to_T_kernel<T>, gS, h + nb, s));
      const int64_t nseg = (int64_t)P.seg_cols.size();
      const int64_t* inst = (const int64_t*)C.seg_inst.ptr;
      qrkit_status rc = banded_tri_solve(ctx, nseg, inst, C.RwS.ptr, V.w, h + nb, true);
      if (rc != QRKIT_OK) return rc;
      rc = banded_tri_solve(ctx, nseg, inst, C.RwS.ptr, V.w, h + nb, false);
      if (rc != QRKIT_OK) return rc;
      LAUNCH(ctx, chain_launch(st, blocks_for(s, 128), 128, 0, axpy_kernel<T>, x + nb, h + nb, s));
    }
    if (V.coupled == QRKIT_COUPLED_DENSE) {
      // dp_S = R_S^{-1} R_S^{-T} (g_S - R12^T h_B), added to p_S and kept in h for the blocks
      if ((rc = dense_normal<T>(ctx, RS, ldRS, s, gS, h + nb, x + nb)) != QRKIT_OK) return rc;
    }
    // dp_B = R_B^{-1} (h_B - R12 dp_S), accumulated into p
    if ((rc = launch_block_backsub<T>(ctx, true, V, O, (const T*)h, s ? h + nb : nullptr, x, 1)) != QRKIT_OK) return rc;
  }
  return QRKIT_OK;
}

qrkit_status composed_factor(qrkit_ctx* ctx, const void* J, const void* S, const void* D, double lambda) {
  if (ctx->precision == QRKIT_FP64) return factor_typed<double>(ctx, J, S, D, lambda);
  return factor_typed<float>(ctx, J, S, D, lambda);
}

template <typename T>
ComposedView<T> composed_view(qrkit_ctx* ctx, const void* J, const void* S) {
  return view<T>(ctx, J, S);
}
template ComposedView<float> composed_view<float>(qrkit_ctx*, const void*, const void*);
template ComposedView<double> composed_view<double>(qrkit_ctx*, const void*, const void*);

qrkit_status composed_column_norms(qrkit_ctx* ctx, const void* J, const void* S, double* D) {
  if (ctx->precision == QRKIT_FP64) return norms_typed<double>(ctx, view<double>(ctx, J, S), D, false);
  return norms_typed<float>(ctx, view<float>(ctx, J, S), D, false);
}

qrkit_status composed_factor_scaled(qrkit_ctx* ctx, const void* J, const void* S, const double* E, bool sorted) {
  if (ctx->precision == QRKIT_FP64) return factor_typed<double>(ctx, J, S, E, 1.0, true, sorted);
  return factor_typed<float>(ctx, J, S, E, 1.0, true, sorted);
}

qrkit_status composed_sort_blocks(qrkit_ctx* ctx, bool* done) {
  Composed& C = ctx->comp;
  *done = C.bins;
  if (!C.bins) return QRKIT_OK;
  return block_sort(ctx, C.bsort, (const int32_t*)ctx->plan.d_start.ptr, (int*)C.hist.ptr, C.bsort_hist,
                    (int32_t*)C.colptr.ptr, (int32_t*)C.bpos.ptr, (int32_t*)C.bord.ptr);
}

qrkit_status composed_window_sums(qrkit_ctx* ctx, const void* S, double* sq) {
  QRKIT_CUDA_TRY(ctx, cudaMemsetAsync(sq, 0, (size_t)ctx->plan.s.shared_cols * sizeof(double), ctx->stream));
  if (ctx->precision == QRKIT_FP64)
    return window_square_sums<double>(ctx, window_sums<double>(ctx, view<double>(ctx, nullptr, S), sq));
  return window_square_sums<float>(ctx, window_sums<float>(ctx, view<float>(ctx, nullptr, S), sq));
}

qrkit_status composed_solve(qrkit_ctx* ctx, bool chained, const void* J, const void* S, const void* b, void* p,
                            int refine_steps) {
  if (ctx->precision == QRKIT_FP64) return solve_typed<double>(ctx, chained, J, S, b, p, refine_steps, false, nullptr);
  const int steps = ctx->precision == QRKIT_FP32 ? 0 : refine_steps;
  return solve_typed<float>(ctx, chained, J, S, b, p, steps, false, nullptr);
}

qrkit_status composed_apply_qt(qrkit_ctx* ctx, const void* b, void* qtb) {
  if (ctx->precision == QRKIT_FP64) return solve_typed<double>(ctx, false, nullptr, nullptr, b, nullptr, 0, true, qtb);
  return solve_typed<float>(ctx, false, nullptr, nullptr, b, nullptr, 0, true, qtb);
}

}  // namespace qrkit

namespace qrkit {

__global__ void multiples_kernel(int64_t* out, int64_t n, int64_t step) {
  dev::chain_wait();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) out[i] = i * step;
}

static qrkit_status upload_i64(qrkit_ctx* ctx, DevBuf& buf, const std::vector<int64_t>& v, const char* what) {
  qrkit_status rc = ensure(ctx, buf, v.size() * sizeof(int64_t), what);
  if (rc != QRKIT_OK) return rc;
  QRKIT_CUDA_TRY(ctx, cudaMemcpy(buf.ptr, v.data(), v.size() * sizeof(int64_t), cudaMemcpyHostToDevice));
  return QRKIT_OK;
}

qrkit_status widen_to_double(qrkit_ctx* ctx, const float* in, double* out, int64_t n) {
  start_launch(ctx->stream, blocks_for(n, 256), 256, 0, widen_kernel, in, out, n);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}

static void release_levels(std::vector<TsqrLevel>& LV) {
  for (auto& L : LV) { release(L.X); release(L.tau); release(L.rhs); release(L.T); }
  LV.clear();
}

void release_composed(Composed& C) {
  release(C.D); release(C.sq); release(C.Fa); release(C.tau); release(C.R12); release(C.ctop);
  release(C.g); release(C.h); release(C.dref);
  release(C.Xw); release(C.Xstart); release(C.rhs_red); release(C.RwS); release(C.cS);
  release(C.res2); release(C.meta); release(C.dense_ws);
  release(C.sort_tab); release(C.hist); release(C.spos); release(C.order); release(C.Xw_s);
  release(C.Xstart_s); release(C.rhs_s); release(C.seg_inst);
  release(C.bs_tab); release(C.bs_colseg); release(C.colptr); release(C.bpos); release(C.bord); release(C.wres);
  release_cr(C.cr);
  release(C.nrm_D); release(C.nrm_L); release(C.nrm_W); release(C.nrm_y); release(C.nrm_As);
  release(C.nrm_rs); release(C.nrm_seg);
  release(C.d_aug_off_d); release(C.d_aug_off_u); release(C.d_red_off_d); release(C.d_red_off_u);
  release_levels(C.levels);
  for (auto& Pn : C.panels) release_levels(Pn.levels);
  release(C.Rs); release(C.cs);
  C = Composed();
}

// Reduced-row offsets per block (host) with / without damping rows.
static std::vector<int64_t> reduced_offsets(const Plan& P, bool damp) {
  std::vector<int64_t> r(P.K + 1, 0);
  for (int64_t i = 0; i < P.K; ++i) r[i + 1] = r[i] + (damp ? P.n[i] : P.n[i] - P.m[i]);
  return r;
}

// Offsets of the augmented blocks for both damping states, the factor buffers, and the
// TSQR level geometry of the dense reduced block.
qrkit_status composed_layout(qrkit_ctx* ctx, size_t elem) {
  Plan& P = ctx->plan;
  Composed& C = ctx->comp;
  qrkit_status rc;
  if (!C.d_aug_off_d.ptr && P.uniform) {
    // blocks of one shape: the offsets are multiples, written on the device
    const int64_t n = P.max_n, m = P.max_m, K = P.K;
    const int64_t step[4] = {(n + m) * m, n * m, n, n - m};
    DevBuf* buf[4] = {&C.d_aug_off_d, &C.d_aug_off_u, &C.d_red_off_d, &C.d_red_off_u};
    for (int q = 0; q < 4; ++q) {
      if ((rc = ensure(ctx, *buf[q], (size_t)(K + 1) * sizeof(int64_t), "block offsets")) != QRKIT_OK) return rc;
      start_launch(ctx->stream, blocks_for(K + 1, 256), 256, 0, multiples_kernel, (int64_t*)buf[q]->ptr, K + 1,
                   step[q]);
      ctx->launches += 1;
      QRKIT_CUDA_TRY(ctx, cudaGetLastError());
    }
    C.aug_values_d = K * step[0]; C.aug_values_u = K * step[1];
    C.red_rows_d = K * step[2]; C.red_rows_u = K * step[3];
  } else if (!C.d_aug_off_d.ptr) {
    std::vector<int64_t> ad(P.K + 1), au(P.K + 1), rd(P.K + 1), ru(P.K + 1);
    ad[0] = au[0] = rd[0] = ru[0] = 0;
    for (int64_t i = 0; i < P.K; ++i) {
      const int64_t n = P.n[i], m = P.m[i];
      ad[i + 1] = ad[i] + (n + m) * m;
      au[i + 1] = au[i] + n * m;
      rd[i + 1] = rd[i] + n;
      ru[i + 1] = ru[i] + (n - m);
    }
    C.aug_values_d = ad[P.K]; C.aug_values_u = au[P.K];
    C.red_rows_d = rd[P.K]; C.red_rows_u = ru[P.K];
    if ((rc = upload_i64(ctx, C.d_aug_off_d, ad, "aug offsets")) != QRKIT_OK) return rc;
    if ((rc = upload_i64(ctx, C.d_aug_off_u, au, "aug offsets")) != QRKIT_OK) return rc;
    if ((rc = upload_i64(ctx, C.d_red_off_d, rd, "reduced offsets")) != QRKIT_OK) return rc;
    if ((rc = upload_i64(ctx, C.d_red_off_u, ru, "reduced offsets")) != QRKIT_OK) return rc;
  }
  if (C.damp && P.first_tall_aug >= 0)
    return fail(ctx, QRKIT_EUNSUPPORTED, "block " + std::to_string(P.first_tall_aug) +
                ": with damping rows the augmented block exceeds 16 rows");
  if (!C.damp && P.first_wide >= 0)
    return fail(ctx, QRKIT_EINVAL, "block " + std::to_string(P.first_wide) +
                " has fewer rows than columns and lambda = 0");
  C.red_rows = C.damp ? C.red_rows_d : C.red_rows_u;
  const int64_t aug = C.damp ? C.aug_values_d : C.aug_values_u;
  {
    const int64_t N = P.cols + P.s.shared_cols;
    if ((rc = ensure(ctx, C.g, (size_t)N * sizeof(double), "refinement g")) != QRKIT_OK) return rc;
    if ((rc = ensure(ctx, C.h, (size_t)N * elem, "refinement h")) != QRKIT_OK) return rc;
  }
  const int s = (int)P.s.shared_cols;
  const int w = P.s.coupled_kind == QRKIT_COUPLED_DENSE ? s : P.s.window;
  if ((rc = ensure(ctx, C.Fa, (size_t)aug * elem, "factor")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.tau, (size_t)P.cols * elem, "tau")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.ctop, (size_t)P.cols * elem, "c")) != QRKIT_OK) return rc;
  if (P.s.coupled_kind != QRKIT_COUPLED_NONE)
    if ((rc = ensure(ctx, C.R12, (size_t)P.cols * w * elem, "R12")) != QRKIT_OK) return rc;
  if (P.s.coupled_kind == QRKIT_COUPLED_WINDOW) {
    // the reduced rows form a banded matrix (rows sorted by window start); its QR runs with
    // the right-hand side in qrkit_solve (the banded solver does not keep Q)
    const int64_t Mr = C.red_rows > 0 ? C.red_rows : 1;
    const int64_t nseg = (int64_t)P.seg_cols.size();
    // blocks of one shape and a parallel banded QR of the segments: the blocks are sorted
    C.bins = P.uniform && w <= 8 && C.red_rows > 0 && P.K < ((int64_t)1 << 31) && (int64_t)s < ((int64_t)1 << 31);
    if (!C.bins) {
      if ((rc = ensure(ctx, C.Xw, (size_t)Mr * w * elem, "reduced rows")) != QRKIT_OK) return rc;
      if ((rc = ensure(ctx, C.Xstart, (size_t)Mr * sizeof(int64_t), "reduced row starts")) != QRKIT_OK) return rc;
      if ((rc = ensure(ctx, C.rhs_red, (size_t)Mr * elem, "reduced rhs")) != QRKIT_OK) return rc;
      if ((rc = ensure(ctx, C.spos, (size_t)Mr * sizeof(int64_t), "reduced row order")) != QRKIT_OK) return rc;
      if ((rc = ensure(ctx, C.order, (size_t)Mr * sizeof(int64_t), "reduced row order")) != QRKIT_OK) return rc;
      if ((rc = ensure(ctx, C.Xstart_s, (size_t)Mr * sizeof(int64_t), "sorted row starts")) != QRKIT_OK) return rc;
    } else {
      if ((rc = ensure(ctx, C.colptr, (size_t)(s + 1) * sizeof(int32_t), "block sort")) != QRKIT_OK) return rc;
      if ((rc = ensure(ctx, C.bpos, (size_t)P.K * sizeof(int32_t), "block sort")) != QRKIT_OK) return rc;
      if ((rc = ensure(ctx, C.bord, (size_t)P.K * sizeof(int32_t), "block sort")) != QRKIT_OK) return rc;
      const size_t rv = (size_t)window_residual_values(P.max_n, P.max_m, elem);
      if ((rc = ensure(ctx, C.wres, rv * P.rows * elem, "refinement residual")) != QRKIT_OK) return rc;
    }
    if ((rc = ensure(ctx, C.RwS, (size_t)s * w * elem, "reduced R")) != QRKIT_OK) return rc;
    if ((rc = ensure(ctx, C.cS, (size_t)s * elem, "reduced c")) != QRKIT_OK) return rc;
    if ((rc = ensure(ctx, C.res2, sizeof(double) * nseg, "reduced residual")) != QRKIT_OK) return rc;
    if ((rc = ensure(ctx, C.Xw_s, (size_t)Mr * w * elem, "sorted reduced rows")) != QRKIT_OK) return rc;
    if ((rc = ensure(ctx, C.rhs_s, (size_t)Mr * elem, "sorted reduced rhs")) != QRKIT_OK) return rc;
    if (C.sort_damp != (C.damp ? 1 : 0)) {
      // chunk tables of the device row sort and the segments' banded instances (host, once
      // per damping state: the reduced rows per block differ with and without damping rows)
      const std::vector<int64_t> ro = reduced_offsets(P, C.damp);
      std::vector<int64_t> c_row0, c_rows, c_hoff, c_col0, c_cols, c_out0, seg_chunk0(nseg + 1, 0);
      std::vector<int64_t> inst(4 * nseg);
      int64_t hoff = 0;
      for (int64_t k = 0; k < nseg; ++k) {
        const int64_t r0 = ro[P.seg_blk0[k]], r1 = ro[P.seg_blk0[k + 1]];
        const int64_t rows = r1 - r0;
        if (rows >= ((int64_t)1 << 31))
          return fail(ctx, QRKIT_EUNSUPPORTED, "a segment has more than 2^31 reduced rows");
        int64_t per = std::max<int64_t>(2048, (rows + 255) / 256);
        seg_chunk0[k] = (int64_t)c_row0.size();
        for (int64_t q = r0; q < r1; q += per) {
          c_row0.push_back(q);
          c_rows.push_back(std::min(per, r1 - q));
          c_hoff.push_back(hoff);
          c_col0.push_back(P.seg_col0[k]);
          c_cols.push_back(P.seg_cols[k]);
          c_out0.push_back(r0);
          hoff += P.seg_cols[k];
        }
        inst[k] = P.seg_cols[k];
        inst[nseg + k] = P.seg_col0[k];
        inst[2 * nseg + k] = r0;
        inst[3 * nseg + k] = rows;
      }
      seg_chunk0[nseg] = (int64_t)c_row0.size();
      if (hoff > ((int64_t)1 << 28))
        return fail(ctx, QRKIT_EUNSUPPORTED, "segments too wide for the device row sort");
      const int64_t nc = (int64_t)c_row0.size();
      std::vector<int64_t> tab;
      for (auto* v : {&c_row0, &c_rows, &c_hoff, &c_col0, &c_cols, &c_out0}) tab.insert(tab.end(), v->begin(), v->end());
      tab.insert(tab.end(), seg_chunk0.begin(), seg_chunk0.end());
      if (!C.bins && (rc = upload_i64(ctx, C.sort_tab, tab, "row sort tables")) != QRKIT_OK) return rc;
      if ((rc = upload_i64(ctx, C.seg_inst, inst, "segment instances")) != QRKIT_OK) return rc;
      if (w <= 8) {
        std::vector<int64_t> ic(inst.begin(), inst.begin() + nseg), i0(inst.begin() + nseg, inst.begin() + 2 * nseg),
            r0v(inst.begin() + 2 * nseg, inst.begin() + 3 * nseg), rv(inst.begin() + 3 * nseg, inst.end());
        if ((rc = cr_build(ctx, C.cr, ic, i0, r0v, rv)) != QRKIT_OK) return rc;
      }
      if (C.bins && !C.bs_tab.ptr) {
        // block sort: chunks of at least 256 blocks, and of an eighth of the segment's columns, which bounds the
        // histograms by 8 counters per block
        std::vector<int64_t> blk0, cseg, chunk0(nseg + 1), hoff(nseg + 1, 0);
        std::vector<int32_t> col_seg((size_t)s);
        for (int64_t k = 0; k < nseg; ++k) {
          const int64_t per = std::max<int64_t>(256, P.seg_cols[k] / 8);
          chunk0[k] = (int64_t)blk0.size();
          for (int64_t q = P.seg_blk0[k]; q < P.seg_blk0[k + 1]; q += per) {
            blk0.push_back(q);
            cseg.push_back(k);
          }
          hoff[k + 1] = hoff[k] + ((int64_t)blk0.size() - chunk0[k]) * P.seg_cols[k];
          std::fill(col_seg.begin() + P.seg_col0[k], col_seg.begin() + P.seg_col0[k] + P.seg_cols[k], (int32_t)k);
        }
        chunk0[nseg] = (int64_t)blk0.size();
        const int64_t nch = (int64_t)blk0.size();
        blk0.push_back(P.K);
        std::vector<int64_t> tab;
        for (auto* v : {&blk0, &cseg, &P.seg_blk0, &P.seg_col0, &chunk0, &hoff}) tab.insert(tab.end(), v->begin(), v->end());
        if ((rc = upload_i64(ctx, C.bs_tab, tab, "block sort tables")) != QRKIT_OK) return rc;
        if ((rc = ensure(ctx, C.bs_colseg, col_seg.size() * sizeof(int32_t), "block sort tables")) != QRKIT_OK) return rc;
        QRKIT_CUDA_TRY(ctx, cudaMemcpy(C.bs_colseg.ptr, col_seg.data(), col_seg.size() * sizeof(int32_t),
                                       cudaMemcpyHostToDevice));
        C.bsort_hist = hoff[nseg];
        if ((rc = ensure(ctx, C.hist, (size_t)std::max<int64_t>(C.bsort_hist, 1) * sizeof(int), "block sort")) != QRKIT_OK)
          return rc;
        const int64_t* t = (const int64_t*)C.bs_tab.ptr;
        C.bsort.num_chunks = nch;
        C.bsort.chunk_blk0 = t;
        C.bsort.chunk_seg = t + (nch + 1);
        C.bsort.seg_blk0 = t + (2 * nch + 1);
        C.bsort.seg_col0 = C.bsort.seg_blk0 + (nseg + 1);
        C.bsort.seg_chunk0 = C.bsort.seg_col0 + (nseg + 1);
        C.bsort.seg_hoff = C.bsort.seg_chunk0 + (nseg + 1);
        C.bsort.col_seg = (const int32_t*)C.bs_colseg.ptr;
      }
      if (!C.bins) {
        // histograms, then one bin total per shared column (the scan's second pass)
        if ((rc = ensure(ctx, C.hist, (size_t)std::max<int64_t>(hoff + P.s.shared_cols, 1) * sizeof(int),
                         "row sort histograms")) != QRKIT_OK)
          return rc;
        const int64_t* t = (const int64_t*)C.sort_tab.ptr;
        C.sort.num_chunks = nc;
        C.sort.chunk_row0 = t;
        C.sort.chunk_rows = t + nc;
        C.sort.chunk_hoff = t + 2 * nc;
        C.sort.chunk_col0 = t + 3 * nc;
        C.sort.chunk_cols = t + 4 * nc;
        C.sort.chunk_out0 = t + 5 * nc;
        C.sort.seg_chunk0 = t + 6 * nc;
        C.sort_hist_entries = hoff;
      }
      C.sort_damp = C.damp ? 1 : 0;
    }
  }
  if (P.s.coupled_kind == QRKIT_COUPLED_DENSE) {
    // float, s a multiple of 32 above 32: column panels of kPanelCols, each a TSQR of its own,
    // their trailing updates on the tensor cores; otherwise one TSQR of CUDA-core tiles (s <= 64)
    const bool panels = elem == sizeof(float) && s > kPanelCols && s <= kMaxDenseS && s % 32 == 0;
    if (s > 64 && !panels)
      return fail(ctx, QRKIT_EUNSUPPORTED,
                  "dense shared block: s <= 64, or (float) s a multiple of 32 up to 512");
    int64_t M0 = C.red_rows + (C.damp ? s : 0);
    if (M0 < s) return fail(ctx, QRKIT_EINVAL, "reduced shared block has fewer rows than columns");
    if (elem == sizeof(float) &&
        (rc = ensure(ctx, C.dref, dense_refine_bytes(P.rows, P.cols, s), "refinement sums")) != QRKIT_OK)
      return rc;
    C.tile_rows = tsqr_rows(ctx, M0, s);
    const int tr = panels ? kPanelRows : C.tile_rows;
    if (panels) M0 = (M0 + 3) & ~int64_t(3);   // zero rows: every row count below is then a multiple of 4
    // the TSQR levels of a panel of pw columns over M rows, w columns wide (panel + trailing);
    // each level's leading dimension is padded to 16 bytes, and the rows that leave a panel
    // (all but its R rows) are laid out level by level, tile by tile, for the next panel
    auto build_levels = [&](std::vector<TsqrLevel>& LV, int64_t M, int pw, int w) -> qrkit_status {
      std::vector<int64_t> Ms;
      while (true) {
        Ms.push_back(M);
        const int64_t tiles = (M + tr - 1) / tr;
        if (tiles <= 1) break;
        const int64_t last = M - (tiles - 1) * tr;
        M = (tiles - 1) * pw + std::min<int64_t>(last, pw);
      }
      if (LV.size() != Ms.size()) {
        release_levels(LV);
        LV.assign(Ms.size(), TsqrLevel());
      }
      int64_t down = 0;
      qrkit_status rc2;
      for (size_t l = 0; l < Ms.size(); ++l) {
        TsqrLevel& L = LV[l];
        L.M = Ms[l];
        L.ld = (L.M + 3) & ~int64_t(3);
        L.tiles = (L.M + tr - 1) / tr;
        L.down0 = down;
        down += L.M - (l + 1 < Ms.size() ? Ms[l + 1] : (int64_t)pw);
        if ((rc2 = ensure(ctx, L.X, (size_t)L.ld * w * elem, "reduced block")) != QRKIT_OK) return rc2;
        if ((rc2 = ensure(ctx, L.rhs, (size_t)L.ld * elem, "reduced rhs")) != QRKIT_OK) return rc2;
        if ((rc2 = ensure(ctx, L.tau, (size_t)L.tiles * pw * (panels ? pw : 1) * elem, "reduced tau")) != QRKIT_OK)
          return rc2;
        if (panels && (rc2 = ensure(ctx, L.T, (size_t)L.tiles * pw * pw * elem, "reduced T")) != QRKIT_OK) return rc2;
      }
      return QRKIT_OK;
    };
    if ((rc = build_levels(C.levels, M0, panels ? kPanelCols : s, s)) != QRKIT_OK) return rc;
    if (panels) {
      const int np = s / kPanelCols;
      if ((int)C.panels.size() != np - 1) {
        for (auto& Pn : C.panels) release_levels(Pn.levels);
        C.panels.assign(np - 1, TsqrPanel());
      }
      for (int j = 1; j < np; ++j) {
        TsqrPanel& Pn = C.panels[j - 1];
        Pn.c0 = j * kPanelCols;
        if ((rc = build_levels(Pn.levels, M0 - Pn.c0, kPanelCols, s - Pn.c0)) != QRKIT_OK) return rc;
      }
      if ((rc = ensure(ctx, C.Rs, (size_t)s * s * elem, "R_S")) != QRKIT_OK) return rc;
      if ((rc = ensure(ctx, C.cs, (size_t)s * elem, "R_S rhs")) != QRKIT_OK) return rc;
    } else {
      for (auto& Pn : C.panels) release_levels(Pn.levels);
      C.panels.clear();
    }
  } else {
    release_levels(C.levels);
    for (auto& Pn : C.panels) release_levels(Pn.levels);
    C.panels.clear();
  }
  return QRKIT_OK;
}

template <typename T>
static qrkit_status solve_r_typed(qrkit_ctx* ctx, const void* qtb, void* p) {
  Plan& P = ctx->plan;
  if (P.s.coupled_kind == QRKIT_COUPLED_WINDOW)
    return fail(ctx, QRKIT_EUNSUPPORTED, "R of a windowed structure is formed in qrkit_solve");
  Composed& C = ctx->comp;
  ComposedView<T> V = view<T>(ctx, nullptr, nullptr);
  FactorOut<T> O = fout<T>(ctx);
  const int s = V.s;
  const T* c = (const T*)qtb;
  T* x = (T*)p;
  if (V.coupled == QRKIT_COUPLED_DENSE) {
    const TsqrLevel& top = C.levels.back();
    const bool pan = !C.panels.empty();
    qrkit_status rc = dense_backsub<T>(ctx, false, pan ? (const T*)C.Rs.ptr : (const T*)top.X.ptr, pan ? s : top.ld, s,
                                       c + P.cols, x + P.cols);
    if (rc != QRKIT_OK) return rc;
  }
  return launch_block_backsub<T>(ctx, V.coupled == QRKIT_COUPLED_DENSE, V, O, c, s ? x + P.cols : nullptr, x, 0);
}

qrkit_status composed_solve_r(qrkit_ctx* ctx, const void* qtb, void* p) {
  if (ctx->precision == QRKIT_FP64) return solve_r_typed<double>(ctx, qtb, p);
  return solve_r_typed<float>(ctx, qtb, p);
}

// Distributed pieces (a dense S whose rows are split over several contexts): the squared column
// sums of J, the R of the reduced shared block, and the block unknowns for given shared ones.
qrkit_status composed_column_sumsq(qrkit_ctx* ctx, const void* J, const void* S, double* out) {
  Composed& C = ctx->comp;
  const int64_t N = ctx->plan.cols + ctx->plan.s.shared_cols;
  qrkit_status rc;
  if ((rc = ensure(ctx, C.D, (size_t)N * sizeof(double), "D")) != QRKIT_OK) return rc;
  if ((rc = composed_column_norms(ctx, J, S, (double*)C.D.ptr)) != QRKIT_OK) return rc;
  QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(out, C.sq.ptr, (size_t)N * sizeof(double), cudaMemcpyDeviceToDevice,
                                      ctx->stream));
  return QRKIT_OK;
}

template <typename T>
__global__ void norms_from_sumsq_kernel(const double* sq, T* D, int64_t n) {
  dev::chain_wait();
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= n) return;
  const double d = sqrt(sq[j]);
  D[j] = (T)(d == 0.0 ? 1.0 : d);   // zero column norm -> 1
}

qrkit_status composed_norms_from_sumsq(qrkit_ctx* ctx, const double* sq, int64_t n, void* D) {
  if (ctx->precision == QRKIT_FP64)
    LAUNCH(ctx, start_launch(ctx->stream, blocks_for(n, 256), 256, 0, norms_from_sumsq_kernel<double>, sq, (double*)D,
                             n));
  else
    LAUNCH(ctx, start_launch(ctx->stream, blocks_for(n, 256), 256, 0, norms_from_sumsq_kernel<float>, sq, (float*)D,
                             n));
  return QRKIT_OK;
}

template <typename T>
__global__ void copy_upper_kernel(const T* X, int64_t ld, int s, T* R) {
  dev::chain_wait();
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)s * s) return;
  const int i = (int)(e % s), j = (int)(e / s);
  R[e] = i <= j ? X[(int64_t)j * ld + i] : T(0);
}

qrkit_status composed_reduced_r(qrkit_ctx* ctx, void* R) {
  Composed& C = ctx->comp;
  const int s = (int)ctx->plan.s.shared_cols;
  const TsqrLevel& top = C.levels.back();
  const void* src = C.panels.empty() ? top.X.ptr : C.Rs.ptr;
  const int64_t ld = C.panels.empty() ? top.ld : s;
  if (ctx->precision == QRKIT_FP64)
    LAUNCH(ctx, start_launch(ctx->stream, blocks_for((int64_t)s * s, 256), 256, 0, copy_upper_kernel<double>,
                             (const double*)src, ld, s, (double*)R));
  else
    LAUNCH(ctx, start_launch(ctx->stream, blocks_for((int64_t)s * s, 256), 256, 0, copy_upper_kernel<float>,
                             (const float*)src, ld, s, (float*)R));
  return QRKIT_OK;
}

template <typename T>
static qrkit_status solve_blocks_typed(qrkit_ctx* ctx, const void* qtb, void* p) {
  Plan& P = ctx->plan;
  ComposedView<T> V = view<T>(ctx, nullptr, nullptr);
  FactorOut<T> O = fout<T>(ctx);
  T* x = (T*)p;
  return launch_block_backsub<T>(ctx, false, V, O, (const T*)qtb, V.s ? x + P.cols : nullptr, x, 0);
}

qrkit_status composed_solve_blocks(qrkit_ctx* ctx, const void* qtb, void* p) {
  if (ctx->precision == QRKIT_FP64) return solve_blocks_typed<double>(ctx, qtb, p);
  return solve_blocks_typed<float>(ctx, qtb, p);
}

}  // namespace qrkit
