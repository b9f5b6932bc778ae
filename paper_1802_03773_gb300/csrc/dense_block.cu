// Q_i^T applied to the coupled columns of a dense S (Sec. 4.2): top rows to R12, the others to the
// reduced shared block.
//
// S (column-major) is read and the reduced block written once, R12 written once; the reflectors are
// a few values per block.  The rows of a CTA's blocks are contiguous in S and in the reduced block,
// so a CTA moves them as whole column segments through shared memory, coalesced for any block
// heights, the next columns arriving (cp.async) while the current ones are transformed; a thread
// per block applies its reflectors to its rows of CC columns in registers.  Bound by HBM and, below
// it, by the three barriers per group of columns.  100,000 blocks 4 x 2, s = 512 (2.05 GB): 457 us,
// 4.5 TB/s; a thread per block reading S itself took 1.54 ms.  14-camera bundle adjustment (blocks of
// 4-12 rows, s = 128): 334 us + 46 us for the factors, against 2.42 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "chain.cuh"
#include "device_util.cuh"
#include "internal.h"

namespace qrkit {
namespace {

constexpr int kThreads = 128;   // blocks per CTA

template <int BYTES>
__device__ __forceinline__ void cp_async_small(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dev::smem_u32(dst)), "l"(src), "n"(BYTES) : "memory");
}

// Blocks of at most NA augmented rows and MM columns, CC columns of S at a time.
template <typename T, int NA, int MM, int CC>
__global__ void __launch_bounds__(kThreads) dense_apply_kernel(ComposedView<T> V, FactorOut<T> O, int cols_per_cta,
                                                               int ldr) {
  dev::chain_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf = reinterpret_cast<T*>(smem_raw);   // two buffers of CC columns x ldr rows
  const int tid = threadIdx.x;
  const int64_t i0 = (int64_t)blockIdx.x * kThreads;
  const int64_t i1 = i0 + kThreads < V.K ? i0 + kThreads : V.K;
  const int64_t ra = V.row_off[i0], rows = V.row_off[i1] - ra;      // S rows of the CTA's blocks
  const int64_t oa = O.red_off[i0], orows = O.red_off[i1] - oa;     // their reduced rows
  const int64_t i = i0 + tid;
  const bool act = i < i1;
  const int n = act ? V.n[i] : 0, m = act ? V.m[i] : 0;
  const int na = act ? n + (O.damp ? m : 0) : 0;
  const int lr = act ? (int)(V.row_off[i] - ra) : 0, lo = act ? (int)(O.red_off[i] - oa) : 0;
  const int64_t col0 = act ? V.col_off[i] : 0;
  const T* F = O.Fa + (act ? O.aug_off[i] : 0);
  T tau[MM], v[MM][NA];   // reflectors, below the diagonal
#pragma unroll
  for (int k = 0; k < MM; ++k) {
    tau[k] = k < m ? O.tau[col0 + k] : T(0);
#pragma unroll
    for (int r = 0; r < NA; ++r) v[k][r] = (k < m && r > k && r < na) ? F[k * na + r] : T(0);
  }
  const int c_begin = (int)blockIdx.y * cols_per_cta;
  const int c_end = min(V.s, c_begin + cols_per_cta);
  // 16-byte copies where every column segment starts on a 16-byte boundary
  constexpr int E = 16 / (int)sizeof(T);
  const bool wide_in = (V.rows % E) == 0 && (ra % E) == 0 && (rows % E) == 0 && (reinterpret_cast<uintptr_t>(V.S) & 15) == 0;
  const bool wide_out = (O.ld0 % E) == 0 && (oa % E) == 0 && (orows % E) == 0 && (reinterpret_cast<uintptr_t>(O.X0) & 15) == 0;
  auto fetch = [&](int c0, T* dst) {
    const int cw = min(CC, c_end - c0);
    for (int c = 0; c < cw; ++c) {
      const T* src = V.S + (int64_t)(c0 + c) * V.rows + ra;
      if (wide_in) {
        for (int e = tid; e < (int)rows / E; e += kThreads) dev::cp_async16(dst + c * ldr + E * e, src + E * e);
      } else {
        for (int e = tid; e < (int)rows; e += kThreads) cp_async_small<sizeof(T)>(dst + c * ldr + e, src + e);
      }
    }
  };
  if (c_begin < c_end) fetch(c_begin, buf);
  dev::cp_async_commit();
  int b = 0;
  for (int c0 = c_begin; c0 < c_end; c0 += CC, b ^= 1) {
    T* cur = buf + b * CC * ldr;
    dev::cp_async_wait_all();
    __syncthreads();   // the columns are here, and the other buffer has been stored
    if (c0 + CC < c_end) fetch(c0 + CC, buf + (b ^ 1) * CC * ldr);
    dev::cp_async_commit();
    const int cw = min(CC, c_end - c0);
    T C[CC][NA];
#pragma unroll
    for (int c = 0; c < CC; ++c)
#pragma unroll
      for (int r = 0; r < NA; ++r) C[c][r] = (c < cw && r < n) ? cur[c * ldr + lr + r] : T(0);
#pragma unroll
    for (int k = 0; k < MM; ++k) {
      if (k < m) {
#pragma unroll
        for (int c = 0; c < CC; ++c) {
          // a double column of zeros costs the FP64 unit as much as any other (20,000 blocks of 8 x 8, s = 1: the
          // solve took 268 us with them, 234 without)
          if (sizeof(T) == 8 && c >= cw) break;
          T w = C[c][k];
#pragma unroll
          for (int r = k + 1; r < NA; ++r) w += v[k][r] * C[c][r];
          w *= tau[k];
          C[c][k] -= w;
#pragma unroll
          for (int r = k + 1; r < NA; ++r) C[c][r] -= w * v[k][r];
        }
      }
    }
    if (act) {
#pragma unroll
      for (int k = 0; k < MM; ++k) {
        if (k < m) {
          T* dst = O.R12 + (col0 + k) * (int64_t)V.s + c0;
          if (cw == CC && (V.s % E) == 0) {   // rows of R12, and c0, on a 16-byte boundary
#pragma unroll
            for (int c = 0; c < CC; c += E) {
              if constexpr (sizeof(T) == 4)
                *reinterpret_cast<float4*>(dst + c) = make_float4(C[c][k], C[c + 1][k], C[c + 2][k], C[c + 3][k]);
              else
                *reinterpret_cast<double2*>(dst + c) = make_double2(C[c][k], C[c + 1][k]);
            }
          } else {
#pragma unroll
            for (int c = 0; c < CC; ++c)
              if (c < cw) dst[c] = C[c][k];
          }
        }
      }
    }
    __syncthreads();   // every block's rows are in registers
#pragma unroll
    for (int r = 0; r < NA; ++r)
      if (r >= m && r < na)
#pragma unroll
        for (int c = 0; c < CC; ++c)
          if (c < cw) cur[c * ldr + lo + (r - m)] = C[c][r];
    __syncthreads();
    for (int c = 0; c < cw; ++c) {
      T* dst = O.X0 + (int64_t)(c0 + c) * O.ld0 + oa;
      const T* src = cur + c * ldr;
      if (wide_out) {
        for (int e = tid; e < (int)orows / E; e += kThreads)
          reinterpret_cast<uint4*>(dst)[e] = reinterpret_cast<const uint4*>(src)[e];
      } else {
        for (int e = tid; e < (int)orows; e += kThreads) dst[e] = src[e];
      }
    }
  }
}

template <typename T, int NA, int MM, int CC>
qrkit_status launch_apply(qrkit_ctx* ctx, const ComposedView<T>& V, const FactorOut<T>& O, int max_n) {
  auto k = dense_apply_kernel<T, NA, MM, CC>;
  constexpr int E = 16 / (int)sizeof(T);
  const int ldr = (kThreads * max_n + E - 1) / E * E;   // columns on 16-byte boundaries
  const size_t smem = 2 * (size_t)CC * ldr * sizeof(T);
  if (smem > 48 * 1024)
    QRKIT_CUDA_TRY(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  // enough CTAs for a dozen per SM: the columns are split over them, CC at a time
  const int64_t bx = (V.K + kThreads - 1) / kThreads;
  const int64_t want = std::max<int64_t>(1, (12 * (int64_t)ctx->num_sms + bx - 1) / bx);
  const int groups = (V.s + CC - 1) / CC;
  const int per = (int)((groups + std::min<int64_t>(want, groups) - 1) / std::min<int64_t>(want, groups));
  const dim3 grid((unsigned)bx, (unsigned)((groups + per - 1) / per));
  chain_launch(ctx->stream, grid, kThreads, smem, k, V, O, per * CC, ldr);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}

}  // namespace

template <typename T>
qrkit_status dense_apply_blocks(qrkit_ctx* ctx, const ComposedView<T>& V, const FactorOut<T>& O) {
  const Plan& P = ctx->plan;
  const int na = P.max_n + (O.damp ? P.max_m : 0);
  if (P.max_m == 1 && na <= 3) return launch_apply<T, 3, 1, 8>(ctx, V, O, P.max_n);
  if (P.max_m <= 2 && na <= 6) return launch_apply<T, 6, 2, 8>(ctx, V, O, P.max_n);
  if (P.max_m <= 3) return launch_apply<T, 16, 3, 4>(ctx, V, O, P.max_n);
  return launch_apply<T, 16, 8, 4>(ctx, V, O, P.max_n);
}
template qrkit_status dense_apply_blocks<float>(qrkit_ctx*, const ComposedView<float>&, const FactorOut<float>&);
template qrkit_status dense_apply_blocks<double>(qrkit_ctx*, const ComposedView<double>&, const FactorOut<double>&);

}  // namespace qrkit
