// TSQR of a dense reduced shared block that is not blocked by column panels (s <= 64; Sec. 2): the QR of one
// tile and its Q^T, in the context's precision.
//
// FP64 runs at about 2 multiply-adds per cycle and SM here, so a warp's FP64 instruction holds its quarter
// of the SM for 64 cycles, and a tile of 256 x 30 needs 60 us of that whatever is done around it.  The
// kernel keeps everything else off that unit: columns with their warp (in registers up to 16 columns; from 17 on
// the loop over a warp's column groups, which holds a barrier, is not unrolled and they live in local memory, a stack
// of 128 bytes per thread for 128-row tiles of doubles), one barrier per column, the sums
// of a warp's columns reduced together by a transposed butterfly (1.5 additions per column instead of 5),
// one reciprocal root and one reciprocal per reflector.  Few tiles of up to 32 columns are cut to 128 rows,
// which spreads the work over more SMs.  FP64, 200 blocks 4 x 2 with 30 shared columns (830 rows): factor
// 302 us, Q^T b 63 us, against 378 and 95 us for a tile in shared memory with a warp per column and two
// barriers; 100,000 blocks 2 x 1 with 5 shared columns: 80 and 31 us against 77 and 45 us.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "chain.cuh"
#include "device_util.cuh"
#include "internal.h"
#include "roots.cuh"

namespace qrkit {
namespace {

constexpr int kThreads = 256;   // 8 warps: column j on warp j % 8
constexpr int kWarps = kThreads / 32;

__host__ __device__ constexpr int pow2_ceil(int m) { return m <= 1 ? 1 : 2 * pow2_ceil((m + 1) / 2); }
__host__ __device__ constexpr int log2_exact(int p) { return p <= 1 ? 0 : 1 + log2_exact(p / 2); }

// Sums of M per-lane values over the warp, returned in every lane.  Transposed butterfly: with the values padded to
// P = 2^ceil(log2 M), each stage sends half of the remaining values to the partner lane and keeps the
// other half, so after log2 P stages each lane holds one partial sum (of value lane >> (5 - log2 P));
// plain stages finish the sums, and one broadcast per value returns them.
template <typename T, int M>
__device__ __forceinline__ void warp_sums(T (&v)[M], int lane) {
  constexpr int P = pow2_ceil(M);
  constexpr int S = 5 - log2_exact(P);
  T w[P];
#pragma unroll
  for (int i = 0; i < P; ++i) w[i] = i < M ? v[i] : T(0);
  int d = 16;
#pragma unroll
  for (int h = P / 2; h >= 1; h /= 2, d >>= 1) {
    const bool up = (lane & d) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const T send = up ? w[i] : w[h + i];
      const T keep = up ? w[h + i] : w[i];
      w[i] = keep + __shfl_xor_sync(0xffffffffu, send, d);
    }
  }
#pragma unroll
  for (int e = 0; e < S; ++e) {
    w[0] += __shfl_xor_sync(0xffffffffu, w[0], d);
    d >>= 1;
  }
#pragma unroll
  for (int j = 0; j < M; ++j) v[j] = __shfl_sync(0xffffffffu, w[0], j << S);
}

// Norm, tau and scale of a reflector with pivot alpha and squared norm sq below it (Sec. 2): beta = -sign(alpha)
// norm, tau = (beta - alpha) / beta = 1 + |alpha| / norm, scale = 1 / (alpha - beta).
__device__ __forceinline__ void reflector(double alpha, double sq, double& beta, double& tau, double& scale) {
  const double n2 = fma(alpha, alpha, sq);
  beta = tau = scale = 0.0;
  if (n2 == 0.0) return;
  const double y = rsqrt(n2);
  const double norm = dev::newton_root(n2, y);
  const double a = fabs(alpha);
  beta = alpha >= 0.0 ? -norm : norm;
  tau = fma(a, y, 1.0);
  scale = __drcp_rn(alpha - beta);
}
__device__ __forceinline__ void reflector(float alpha, float sq, float& beta, float& tau, float& scale) {
  const float norm = sqrtf(alpha * alpha + sq);
  beta = tau = scale = 0.f;
  if (norm == 0.f) return;
  beta = alpha >= 0.f ? -norm : norm;
  tau = (beta - alpha) / beta;
  scale = 1.f / (alpha - beta);
}

// One tile of at most 32 RPL rows (`rows` of the level each) and s <= 8 CPW columns: row lane + 32 u on the lane,
// column j on warp j % 8.  At step k the reflector v_k is read from shared memory (two alternating slots) by every
// warp and applied to its columns after k; the warp of column k + 1 forms the next reflector right after updating it.  V below / R
// on and above the diagonal in place, tau to taus[tile s + k], the R rows (zeros below) to the next level.
template <typename T, int RPL, int CPW>
__global__ void __launch_bounds__(kThreads) tsqr_tile_kernel(T* X, int64_t ld, int64_t M, int s, int rows, T* taus,
                                                             T* Xn, int64_t ldn) {
  dev::chain_wait();
  constexpr int kRows = 32 * RPL;
  __shared__ T V[2][kRows];
  __shared__ T tslot[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * rows;
  const int r = (int)(M - r0 < (int64_t)rows ? M - r0 : (int64_t)rows);   // <= 32 RPL
  const int kmax = r < s ? r : s;
  const int mine = sizeof(T) == 8 ? (s - warp + kWarps - 1) / kWarps : CPW;   // the warp's columns, without those of zeros
  T a[CPW][RPL];
#pragma unroll
  for (int i = 0; i < CPW; ++i) {
    const int j = warp + kWarps * i;
    const T* src = X + (int64_t)j * ld + r0 + lane;
#pragma unroll
    for (int u = 0; u < RPL; ++u) a[i][u] = j < s && lane + 32 * u < r ? src[32 * u] : T(0);
  }
  auto form = [&](int k, T (&c)[RPL]) {
    T sq[1] = {T(0)};
    T ak = T(0);
#pragma unroll
    for (int u = 0; u < RPL; ++u) {
      const int i = lane + 32 * u;
      if (i > k) sq[0] += c[u] * c[u];
      if (u == (k >> 5)) ak = c[u];
    }
    warp_sums<T, 1>(sq, lane);
    const T alpha = __shfl_sync(0xffffffffu, ak, k & 31);
    T beta, tau, scale;
    reflector(alpha, sq[0], beta, tau, scale);
#pragma unroll
    for (int u = 0; u < RPL; ++u) {
      const int i = lane + 32 * u;
      if (i > k) c[u] *= scale;
      else if (i == k) c[u] = beta;
      V[k & 1][i] = i > k ? c[u] : (i == k ? T(1) : T(0));
    }
    if (lane == 0) {
      tslot[k & 1] = tau;
      taus[(int64_t)blockIdx.x * s + k] = tau;
    }
  };
  if (warp == 0 && kmax > 0) form(0, a[0]);
#pragma unroll
  for (int i = 0; i < CPW; ++i) {
    for (int w = 0; w < kWarps; ++w) {
      const int k = kWarps * i + w;
      if (k >= kmax) break;
      __syncthreads();   // reflector k is in its slot; the other slot has been read
      const T t = tslot[k & 1];
      T v[RPL], p[CPW];
#pragma unroll
      for (int u = 0; u < RPL; ++u) v[u] = V[k & 1][lane + 32 * u];
      // columns after k: the warp's i' > i, and its i-th if that lies after k
#pragma unroll
      for (int c = 0; c < CPW; ++c) {
        p[c] = T(0);
        if (c < mine && (c > i || (c == i && warp > w))) {
#pragma unroll
          for (int u = 0; u < RPL; ++u) p[c] += v[u] * a[c][u];
        }
      }
      if (i + 1 < mine || (i < mine && warp > w)) {
        T q[CPW];
#pragma unroll
        for (int c = 0; c < CPW; ++c) q[c] = c >= i ? p[c] : T(0);
        warp_sums<T, CPW>(q, lane);
#pragma unroll
        for (int c = 0; c < CPW; ++c) {
          if (c < mine && (c > i || (c == i && warp > w))) {
            const T wt = q[c] * t;
#pragma unroll
            for (int u = 0; u < RPL; ++u) a[c][u] -= wt * v[u];
          }
        }
      }
      if (k + 1 < kmax && (k + 1) % kWarps == warp) {
        if (w + 1 < kWarps) form(k + 1, a[i]);
        else if (i + 1 < CPW) form(k + 1, a[i + 1 < CPW ? i + 1 : i]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < CPW; ++i) {
    const int j = warp + kWarps * i;
    if (j >= s) continue;
    T* dst = X + (int64_t)j * ld + r0 + lane;
#pragma unroll
    for (int u = 0; u < RPL; ++u)
      if (lane + 32 * u < r) dst[32 * u] = a[i][u];
    if (Xn) {
      T* up = Xn + (int64_t)j * ldn + (int64_t)blockIdx.x * s + lane;
#pragma unroll
      for (int u = 0; u < RPL; ++u)
        if (lane + 32 * u < kmax) up[32 * u] = lane + 32 * u <= j ? a[i][u] : T(0);
    }
  }
}

// Q_tile^T applied to a level's right-hand side, reflector by reflector; the top min(r, s) entries go to the next
// level.  Four warps (one per quarter of the SM), RPT rows per thread, the next reflector loaded a step
// ahead; one barrier per reflector: every warp adds the four partial sums itself.
constexpr int kQtThreads = 128;

template <typename T, int RPT>
__global__ void __launch_bounds__(kQtThreads) tsqr_qt_kernel(const T* X, int64_t ld, int64_t M, int s, const T* taus,
                                                             T* rhs, T* rhs_next) {
  dev::chain_wait();
  constexpr int kRows = kQtThreads * RPT;
  __shared__ T part[2][kQtThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * kRows;
  const int r = (int)(M - r0 < (int64_t)kRows ? M - r0 : (int64_t)kRows);
  const int kmax = r < s ? r : s;
  T y[RPT], v[RPT];
  auto fetch = [&](int k, T (&d)[RPT]) {
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const int i = tid + kQtThreads * q;
      d[q] = i > k && i < r ? X[(int64_t)k * ld + r0 + i] : (i == k ? T(1) : T(0));
    }
  };
#pragma unroll
  for (int q = 0; q < RPT; ++q) y[q] = tid + kQtThreads * q < r ? rhs[r0 + tid + kQtThreads * q] : T(0);
  if (kmax > 0) fetch(0, v);
  for (int k = 0; k < kmax; ++k) {
    T nv[RPT];
    const T tau = taus[(int64_t)blockIdx.x * s + k];
    if (k + 1 < kmax) fetch(k + 1, nv);
    T w[1] = {T(0)};
#pragma unroll
    for (int q = 0; q < RPT; ++q) w[0] += v[q] * y[q];
    warp_sums<T, 1>(w, lane);
    if (lane == 0) part[k & 1][warp] = w[0];
    __syncthreads();
    const T wt = ((part[k & 1][0] + part[k & 1][1]) + (part[k & 1][2] + part[k & 1][3])) * tau;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      y[q] -= wt * v[q];
      if (k + 1 < kmax) v[q] = nv[q];
    }
  }
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    const int i = tid + kQtThreads * q;
    if (i < r) rhs[r0 + i] = y[q];
    if (rhs_next && i < kmax) rhs_next[(int64_t)blockIdx.x * s + i] = y[q];
  }
}

// CPW column groups of 8.  A double column of zeros costs the FP64 unit as much as any other, so doubles take as many
// groups as s has (rounded up to the next power of two of groups, s = 33 was 1.1 to 1.4 times as slow over the whole
// solve); floats take the next power of two.
template <typename T, int RPL, int CPW = 1>
void launch_tile(unsigned g, cudaStream_t st, T* X, int64_t ld, int64_t M, int s, int rows, T* taus, T* Xn,
                 int64_t ldn) {
  if constexpr (CPW < 8) {
    if (s > kWarps * CPW)
      return launch_tile<T, RPL, sizeof(T) == 8 ? CPW + 1 : 2 * CPW>(g, st, X, ld, M, s, rows, taus, Xn, ldn);
  }
  chain_launch(st, g, kThreads, 0, (tsqr_tile_kernel<T, RPL, CPW>), X, ld, M, s, rows, taus, Xn, ldn);
}

}  // namespace

int tsqr_rows(const qrkit_ctx* ctx, int64_t M, int s) { return s <= 32 && M <= 128 * (int64_t)ctx->num_sms ? 128 : 256; }

template <typename T>
qrkit_status tsqr_tile(qrkit_ctx* ctx, T* X, int64_t ld, int64_t M, int s, int rows, T* taus, T* Xn, int64_t ldn,
                       int64_t tiles) {
  if (s > 64 || (rows != 128 && rows != 256)) return fail(ctx, QRKIT_EUNSUPPORTED, "TSQR tile: at most 64 columns");
  // a short top level does not walk the rows of a full tile
  const int64_t most = M < rows ? M : rows;
  if (most <= 64) launch_tile<T, 2>((unsigned)tiles, ctx->stream, X, ld, M, s, rows, taus, Xn, ldn);
  else if (most <= 128) launch_tile<T, 4>((unsigned)tiles, ctx->stream, X, ld, M, s, rows, taus, Xn, ldn);
  else launch_tile<T, 8>((unsigned)tiles, ctx->stream, X, ld, M, s, rows, taus, Xn, ldn);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}
template qrkit_status tsqr_tile<float>(qrkit_ctx*, float*, int64_t, int64_t, int, int, float*, float*, int64_t, int64_t);
template qrkit_status tsqr_tile<double>(qrkit_ctx*, double*, int64_t, int64_t, int, int, double*, double*, int64_t,
                                        int64_t);

template <typename T>
qrkit_status tsqr_qt(qrkit_ctx* ctx, const T* X, int64_t ld, int64_t M, int s, int rows, const T* taus, T* rhs,
                     T* rhs_next, int64_t tiles) {
  if (rows == 128)
    chain_launch(ctx->stream, (unsigned)tiles, kQtThreads, 0, (tsqr_qt_kernel<T, 1>), X, ld, M, s, taus, rhs,
                 rhs_next);
  else
    chain_launch(ctx->stream, (unsigned)tiles, kQtThreads, 0, (tsqr_qt_kernel<T, 2>), X, ld, M, s, taus, rhs,
                 rhs_next);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}
template qrkit_status tsqr_qt<float>(qrkit_ctx*, const float*, int64_t, int64_t, int, int, const float*, float*, float*,
                                     int64_t);
template qrkit_status tsqr_qt<double>(qrkit_ctx*, const double*, int64_t, int64_t, int, int, const double*, double*,
                                      double*, int64_t);

}  // namespace qrkit
