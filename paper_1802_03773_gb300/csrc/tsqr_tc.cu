// Column-panel TSQR of the dense reduced shared block (float, s a multiple of 32).
//
// The reduced block is factored by panels of 32 columns (Sec. 2, compact WY): each panel is a TSQR
// over tiles of kPanelRows = 1024 rows.  tsqr_panel_tile_kernel factors a tile (Householder QR with
// the columns in registers, and the tile's compact-WY T); tsqr_panel_apply_kernel applies the tiles'
// Q^T = I - Y T^T Y^T to the later columns; tsqr_panel_qt_kernel does the same for a right-hand side.
//
// Tiles of 1024 rows leave 32 R rows of 1024 for the next level, so 400,000 rows need three levels
// (391, 13 and 1 tiles) where tiles of 256 rows needed five, and a reflector's reductions and
// barriers are paid once per 1024 rows.  100,000 blocks 4 x 2, factor + solve with one refinement
// step, against 256-row tiles with tcgen05 updates: s = 512 37.4 -> 13.0 ms (panel tiles 9.07 -> 2.63,
// updates 21.6 -> 6.34, Q^T b 3.25 -> 0.49), s = 128 5.58 -> 2.30 ms.
//
// Level matrices are column-major with a leading dimension, a row count and row offsets that are
// multiples of 4 (the first level is padded with zero rows), so every access is a 16-byte one.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "chain.cuh"
#include "device_util.cuh"
#include "f32x2.cuh"
#include "internal.h"
#include "roots.cuh"

namespace qrkit {
namespace {

constexpr int kTR = kPanelRows;   // tile rows
constexpr int kNb = kPanelCols;   // panel width
static_assert(kTR == 1024 && kNb == 32, "the kernels' thread layouts");

using dev::f2;
using dev::fma2;
using dev::mul2;
using dev::pack2;
using dev::sum2;
using dev::unpack2;

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// Sum over the warp of 32 values per lane, transposed: lane l ends with the sum over all lanes
// of v[l] (31 shuffles: at each halving a lane keeps the half of the pairs its bit selects).
__device__ __forceinline__ float transpose_reduce(float (&v)[32], int lane) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    const bool upper = (lane & d) != 0;
#pragma unroll
    for (int k = 0; k < d; ++k) {
      const float send = upper ? v[k] : v[k + d];
      const float keep = upper ? v[k + d] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, d);
    }
  }
  return v[0];
}

// Sums over the warp of four values per lane: lane l ends with the sum of v[l >> 3] (6 shuffles).
__device__ __forceinline__ float sum4(const float (&v)[4], int lane) {
  const bool up = (lane & 16) != 0, odd = (lane & 8) != 0;
  float x = up ? v[2] : v[0], y = up ? v[3] : v[1];
  x += __shfl_xor_sync(0xffffffffu, up ? v[0] : v[2], 16);
  y += __shfl_xor_sync(0xffffffffu, up ? v[1] : v[3], 16);
  float z = (odd ? y : x) + __shfl_xor_sync(0xffffffffu, odd ? x : y, 8);
#pragma unroll
  for (int d = 4; d >= 1; d >>= 1) z += __shfl_xor_sync(0xffffffffu, z, d);
  return z;
}

// ---- the QR of one tile (up to 1024 x 32) of a panel ----
//
// 8 warps; columns 4 w .. 4 w + 3 live in the registers of warp w, rows 128 u + 4 lane + q (u < NU, q < 4) on
// the lane.  Every reflector v_k has a place of its own in shared memory and an mbarrier that says it is there, so
// the warps run through k = 0, 1, .. at their own pace without a barrier of the CTA.  Reflectors before a
// warp's columns update them; its own four it forms one after the other straight from its registers; against
// those after them its columns give G[c][k] = v_c^T v_k (v_k is zero above row k, so the R entries above a
// reflector drop out).  Bound by the chain from one reflector to the next.  With one column per warp and turn
// (16 warps, column j on warp j % 16) that was 2,200 cycles: 340 until the next warp saw the reflector, 500 to load
// it beside 15 others, 160 for the product, 200 and 190 for the two reductions, 250 for update and norm, 360 for
// a root and two divisions, 260 to store; with four columns on a warp three of four reflectors skip the first two,
// and one reciprocal root serves norm and tau.  A wave of 1024-row tiles of cold input: 38 us then, 30 us now.
// T comes last, its two diagonal 16 x 16 blocks by a warp each
// (T[k][k] = tau_k, the strict upper part of column k -tau_k T[:, :k] G[:k, k]), then T12 = -T11 G12 T22.
// NU = 2, 4 or 8: the smallest that covers the level's tiles, so that a short top level does not walk 1024 rows.
constexpr int kPT = 256;
constexpr int kPad = kNb + 1;   // row stride of G and T in shared memory (conflict-free columns)
constexpr uint32_t kWaitLimit = 1u << 22;   // polls of a reflector (formed within microseconds)

template <int NU>
constexpr size_t panel_tile_smem() { return (size_t)kNb * 128 * NU * 4; }

template <int NU>
__global__ void __launch_bounds__(kPT, 1)
tsqr_panel_tile_kernel(float* X, int64_t ld, int64_t M, float* Xn, int64_t ldn, float* Tout, float* Gout, int* status) {
  dev::chain_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* V = reinterpret_cast<float*>(smem_raw);   // 32 reflectors of 128 NU rows
  __shared__ float Gs[kNb * kPad], Tm[kNb * kPad], Ws[16 * kPad];
  __shared__ float tau_s[kNb];
  __shared__ __align__(8) uint64_t ready[kNb];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * kTR;
  const int r = (int)(M - r0 < (int64_t)kTR ? M - r0 : (int64_t)kTR);   // a multiple of 4
  const int kmax = r < kNb ? r : kNb;                                   // so this too
  const int c0 = 4 * warp;
  float* x = X + (int64_t)c0 * ld + r0 + 4 * lane;

  f2 a[4][2 * NU];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
      if (128 * u + 4 * lane < r) p = *reinterpret_cast<const float4*>(x + (int64_t)j * ld + 128 * u);
      a[j][2 * u] = pack2(p.x, p.y);
      a[j][2 * u + 1] = pack2(p.z, p.w);
    }
  for (int e = tid; e < kNb * kPad; e += kPT) Gs[e] = Tm[e] = 0.f;
  if (tid < kNb) {
    tau_s[tid] = 0.f;
    dev::mbar_init(&ready[tid], 1);
  }
  dev::fence_mbar_init();
  __syncthreads();

  // the reflector of column k from its register column c: the column below k scaled to v (v_k = 1, stored
  // implicitly), beta on the diagonal; v written to its place and announced; rows 4 lane .. + 3 of v to
  // head, tau returned.
  auto form = [&](int k, f2 (&c)[2 * NU], f2 (&head)[2]) -> float {
    float h[4];   // rows 4 lane .. 4 lane + 3: the only ones that can lie on or above row k
    unpack2(c[0], h[0], h[1]);
    unpack2(c[1], h[2], h[3]);
    f2 s2 = 0ull, s3 = 0ull;
#pragma unroll
    for (int u = 1; u < NU; ++u) {
      s2 = fma2(c[2 * u], c[2 * u], s2);
      s3 = fma2(c[2 * u + 1], c[2 * u + 1], s3);
    }
    float sq = sum2(s2) + sum2(s3), ak = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = 4 * lane + q;
      if (i > k) sq += h[q] * h[q];
      if (i == k) ak = h[q];
    }
    const float alpha = __shfl_sync(0xffffffffu, ak, k >> 2);
    sq = warp_sum(sq);
    const float n2 = fmaf(alpha, alpha, sq);
    const bool some = n2 != 0.f;
    const float seed = rsqrtf(some ? n2 : 1.f);
    const float norm = dev::newton_root(n2, seed), y = dev::newton_inverse(norm, seed);
    const float beta = some ? (alpha >= 0.f ? -norm : norm) : 0.f;
    const float t = some ? fmaf(fabsf(alpha), y, 1.f) : 0.f;        // (beta - alpha) / beta
    const float scale = some ? __frcp_rn(alpha - beta) : 0.f;
    float v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = 4 * lane + q;
      if (i > k) h[q] *= scale;
      else if (i == k) h[q] = beta;
      v[q] = i > k ? h[q] : (i == k ? 1.f : 0.f);
    }
    c[0] = pack2(h[0], h[1]);
    c[1] = pack2(h[2], h[3]);
    head[0] = pack2(v[0], v[1]);
    head[1] = pack2(v[2], v[3]);
    float* dst = V + k * (128 * NU) + 4 * lane;
    *reinterpret_cast<ulonglong2*>(dst) = make_ulonglong2(head[0], head[1]);
    const f2 sc = pack2(scale, scale);
#pragma unroll
    for (int u = 1; u < NU; ++u) {
      c[2 * u] = mul2(c[2 * u], sc);
      c[2 * u + 1] = mul2(c[2 * u + 1], sc);
      *reinterpret_cast<ulonglong2*>(dst + 128 * u) = make_ulonglong2(c[2 * u], c[2 * u + 1]);
    }
    if (lane == 0) tau_s[k] = t;
    __syncwarp();
    if (lane == 0)
      asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(dev::smem_u32(&ready[k])) : "memory");
    return t;
  };
  // products with v (its first two pairs in head, the others in v) and its update of a column
  auto dot = [&](const f2 (&head)[2], const f2 (&v)[2 * NU], const f2 (&c)[2 * NU]) -> float {
    f2 d = 0ull, e = 0ull;
#pragma unroll
    for (int u = 1; u < NU; ++u) {
      d = fma2(v[2 * u], c[2 * u], d);
      e = fma2(v[2 * u + 1], c[2 * u + 1], e);
    }
    d = fma2(head[0], c[0], d);
    e = fma2(head[1], c[1], e);
    return sum2(d) + sum2(e);
  };
  auto update = [&](float w, const f2 (&head)[2], const f2 (&v)[2 * NU], f2 (&c)[2 * NU]) {
    const f2 w2 = pack2(w, w);
    c[0] = fma2(w2, head[0], c[0]);
    c[1] = fma2(w2, head[1], c[1]);
#pragma unroll
    for (int u = 2; u < 2 * NU; ++u) c[u] = fma2(w2, v[u], c[u]);
  };
  f2 v[2 * NU], head[2];
  // waits for reflector k and loads it; false if it did not come
  auto take = [&](int k) -> bool {
    bool here = false;
    for (uint32_t it = 0; it < kWaitLimit && !here; ++it) here = dev::mbar_try_wait(&ready[k], 0u);
    if (!__all_sync(0xffffffffu, here)) return false;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(V + k * (128 * NU) + 128 * u + 4 * lane);
      v[2 * u] = w.x;
      v[2 * u + 1] = w.y;
    }
    head[0] = v[0];
    head[1] = v[1];
    return true;
  };

  bool ok = true;
  for (int k = 0; k < kmax && k < c0; ++k) {
    if (!(ok = take(k))) break;
    const float t = -tau_s[k];
    float p[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) p[j] = dot(head, v, a[j]);
    const float z = sum4(p, lane);
#pragma unroll
    for (int j = 0; j < 4; ++j) update(__shfl_sync(0xffffffffu, z, 8 * j) * t, head, v, a[j]);
  }
  if (ok && c0 < kmax) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float t = -form(c0 + i, a[i], head);
      float p[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) p[j] = j != i ? dot(head, a[i], a[j]) : 0.f;
      const float z = sum4(p, lane);
#pragma unroll
      for (int j = i + 1; j < 4; ++j) update(__shfl_sync(0xffffffffu, z, 8 * j) * t, head, a[i], a[j]);
      if ((lane & 7) == 0 && (lane >> 3) < i) Gs[(c0 + (lane >> 3)) * kPad + c0 + i] = z;
    }
  }
  for (int k = c0 + 4; k < kmax && ok; ++k) {
    if (!(ok = take(k))) break;
    float p[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) p[j] = dot(head, v, a[j]);
    const float z = sum4(p, lane);
    if ((lane & 7) == 0) Gs[(c0 + (lane >> 3)) * kPad + k] = z;
  }
  if (__syncthreads_or(!ok)) {
    if (tid == 0 && status) atomicCAS(status, 0, QRKIT_ETIMEOUT);
    return;
  }
  // V below / R on and above the diagonal in place; the R rows (zeros below) to the next level
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int u = 0; u < NU; ++u)
      if (128 * u + 4 * lane < r)
        *reinterpret_cast<ulonglong2*>(x + (int64_t)j * ld + 128 * u) = make_ulonglong2(a[j][2 * u], a[j][2 * u + 1]);
  if (4 * lane < kmax) {
    const int64_t n0 = (int64_t)blockIdx.x * kNb + 4 * lane;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float h[4];
      unpack2(a[j][0], h[0], h[1]);
      unpack2(a[j][1], h[2], h[3]);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (4 * lane + q > c0 + j) h[q] = 0.f;
      *reinterpret_cast<float4*>(Xn + (int64_t)(c0 + j) * ldn + n0) = make_float4(h[0], h[1], h[2], h[3]);
    }
  }
  // T: warps 0 and 1 the diagonal blocks (lane l < 16 holds row l of the block; sums run over all 16
  // columns, those not yet formed are zero)
  if (warp < 2) {
    const int o = 16 * warp, row = o + (lane & 15);
    float tr[16];   // row `row` of the block
#pragma unroll
    for (int m = 0; m < 16; ++m) tr[m] = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float tk = tau_s[o + k];
      float q0 = 0.f, q1 = 0.f;
#pragma unroll
      for (int m = 0; m < k; ++m) {
        if (m & 1) q1 += tr[m] * Gs[(o + m) * kPad + o + k];
        else q0 += tr[m] * Gs[(o + m) * kPad + o + k];
      }
      tr[k] = (lane & 15) < k ? -(q0 + q1) * tk : ((lane & 15) == k ? tk : 0.f);
    }
    if (lane < 16) {
#pragma unroll
      for (int m = 0; m < 16; ++m) Tm[row * kPad + o + m] = tr[m];
    }
  }
  __syncthreads();
  {   // W = G12 T22
    const int i = tid >> 4, j = tid & 15;
    float w = 0.f;
#pragma unroll
    for (int m = 0; m < 16; ++m) w += Gs[i * kPad + 16 + m] * Tm[(16 + m) * kPad + 16 + j];
    Ws[i * kPad + j] = w;
  }
  __syncthreads();
  {   // T12 = -T11 W
    const int i = tid >> 4, j = tid & 15;
    float w = 0.f;
#pragma unroll
    for (int m = 0; m < 16; ++m) w += Tm[i * kPad + m] * Ws[m * kPad + j];
    Tm[i * kPad + 16 + j] = -w;
  }
  __syncthreads();
  for (int e = tid; e < kNb * kNb; e += kPT) {
    const int m = e / kNb, k = e % kNb;
    Tout[(int64_t)blockIdx.x * (kNb * kNb) + e] = Tm[m * kPad + k];
    Gout[(int64_t)blockIdx.x * (kNb * kNb) + e] = m == k ? tau_s[k] : Gs[m * kPad + k];
  }
}

// ---- a factored panel's tile reflectors applied to the columns after it ----
//
// One CTA takes a tile and a range of the trailing columns C; its two teams of 8 warps take 16
// columns at a time in turn, so that one team's loads and barriers overlap the other's arithmetic.
// A warp holds 128 rows x 16 columns of C in registers, in the fragment layout of
// mma.m16n8k8 (tf32, the columns of C as its rows), which serves both products:
//   W^T = C^T Y      C as the A operand (a permutation of the rows within a group of 16, the same
//                    in both operands, makes a thread's four consecutive rows two k pairs);
//   C^T -= Z^T Y^T   the same registers as the accumulator layout, Z = T^T W.
// The warps' partial W are added through shared memory.  Products are 3xTF32 (x = hi + lo, hi hi +
// hi lo + lo hi) with FP32 accumulation; W is accumulated on the tensor cores over 16 rows at a time
// and then added in FP32, so a sum over 1024 rows is rounded like one of FP32 multiply-adds (a
// 256-row sum by chunks of 16: 1.1e-7 against 3.3e-7 for a chain of fmaf), and the correction is
// subtracted in FP32.  At K = 32 the update does 16 flop per byte of C, so it is bound by memory
// and by the 286 TFLOP/s that mma.sync reaches here about equally; C crosses the chip once and
// never goes through shared memory, which tcgen05 operands in hi and lo halves would need twice.
constexpr int kAT = 512;        // threads: two teams of 8 warps
constexpr int kGC = 16;         // columns per group
constexpr int kPW = 40;         // row stride of the partial W and of Z (conflict-free)

size_t panel_apply_smem() {
  return (size_t)kNb * kTR * 4 + (size_t)kNb * kNb * 4 + 2 * 8 * (size_t)kGC * kPW * 4 + 2 * 2 * (size_t)kGC * kPW * 4;
}

// Shared-memory position of row i of reflector l: bits 3 and 4 of the row flipped by l, which keeps
// both products' reads (16-byte over rows, 8-byte over reflectors) free of bank conflicts.
__device__ __forceinline__ int ypos(int l, int i) { return l * kTR + (i ^ (((l & 1) << 4) | ((l & 2) << 2))); }

// x = h + l for 3xTF32: h rounded to TF32, l = x - h exactly.  l has at most 12 bits, of which the tensor
// core reads the top 11: an error of at most one unit of x's last place, the same as rounding l.
// The rounding is an add and a mask, which issue at twice the rate of cvt.rna.tf32 here; a NaN whose
// mantissa the add overflows still arrives through l.
struct Split {
  uint32_t h, l;
};
__device__ __forceinline__ Split split_tf32(float x) {
  Split s;
  s.h = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  s.l = __float_as_uint(x - __uint_as_float(s.h));
  return s;
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void team_sync(int team) {
  asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(kAT / 2) : "memory");
}

__global__ void __launch_bounds__(kAT, 1)
tsqr_panel_apply_kernel(const float* X, int64_t ld, int64_t M, const float* Tin, int n, int chunk, float* up,
                        int64_t ldu, float* down, int64_t ldd, int64_t down0) {
  dev::chain_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* Y = reinterpret_cast<float*>(smem_raw);   // 32 reflectors x 1024 rows, ypos()
  float* Tm = Y + kNb * kTR;                       // 32 x 32: T[l][i] at l * 32 + i
  float* Pt = Tm + kNb * kNb;                      // partial W per team and warp: [col][reflector]
  float* Zs = Pt + 2 * 8 * kGC * kPW;              // W and Z per team: [col][reflector]

  const int tid = threadIdx.x, lane = tid & 31;
  const int team = tid >> 8, tt = tid & 255, warp = tt >> 5;
  const int kq = lane & 3, nq = lane >> 2;
  const int64_t tile = blockIdx.x;
  const int64_t r0 = tile * kTR;
  const int r = (int)(M - r0 < (int64_t)kTR ? M - r0 : (int64_t)kTR);   // a multiple of 4
  const int kmax = r < kNb ? r : kNb;
  const int j0 = (int)blockIdx.y * chunk;
  const int nc = n - j0 < chunk ? n - j0 : chunk;   // a multiple of 32

  // Y: the stored reflectors, zero past the tile's end
  for (int e = tid; e < kNb * (kTR / 4); e += kAT) {
    const int l = e / (kTR / 4), i = 4 * (e % (kTR / 4));
    float* dst = Y + ypos(l, i);
    if (i < r) dev::cp_async16(dst, X + (int64_t)l * ld + r0 + i);
    else *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  dev::cp_async_commit();
  for (int e = tid; e < kNb * kNb; e += kAT) Tm[e] = Tin[tile * (kNb * kNb) + e];
  dev::cp_async_wait_all();
  __syncthreads();
  // 1 on the diagonal, 0 above it (where R is stored) and for reflectors a short tile lacks
  for (int e = tid; e < kNb * kNb; e += kAT) {
    const int l = e / kNb, i = e % kNb;
    if (i <= l || l >= kmax) Y[ypos(l, i)] = (i == l && l < kmax) ? 1.f : 0.f;
  }
  __syncthreads();

  float* part = Pt + (team * 8 + warp) * (kGC * kPW);
  float* Ws = Zs + team * 2 * (kGC * kPW);
  float* Zt = Ws + kGC * kPW;
  const int wr = 128 * warp;                       // the warp's first row
  for (int g = team; g < nc / kGC; g += 2) {
    const int jc = j0 + g * kGC;
    const float* Cg = X + (int64_t)(kNb + jc + nq) * ld + r0;
    if (g + 2 < nc / kGC)   // the team's next columns on their way into L2
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i = 32 * (tt & 31);
        if (i < r)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(X + (int64_t)(kNb + jc + 2 * kGC + 2 * warp + q) * ld + r0 + i));
      }
    float4 ca[8], cb[8];                           // columns nq and nq + 8, rows wr + 16 G + 4 kq ..
#pragma unroll
    for (int G = 0; G < 8; ++G) {
      const int i = wr + 16 * G + 4 * kq;
      ca[G] = cb[G] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < r) {
        ca[G] = *reinterpret_cast<const float4*>(Cg + i);
        cb[G] = *reinterpret_cast<const float4*>(Cg + 8 * ld + i);
      }
    }
    // W^T = C^T Y over the warp's rows
    float w[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) w[j][q] = 0.f;
    if (wr < r) {
#pragma unroll
      for (int G = 0; G < 8; ++G) {
        const Split ax = split_tf32(ca[G].x), ay = split_tf32(ca[G].y), az = split_tf32(ca[G].z),
                    aw = split_tf32(ca[G].w);
        const Split bx = split_tf32(cb[G].x), by = split_tf32(cb[G].y), bz = split_tf32(cb[G].z),
                    bw = split_tf32(cb[G].w);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 yv = *reinterpret_cast<const float4*>(Y + ypos(8 * j + nq, wr + 16 * G + 4 * kq));
          const Split yx = split_tf32(yv.x), yy = split_tf32(yv.y), yz = split_tf32(yv.z), yw = split_tf32(yv.w);
          float d[4] = {0.f, 0.f, 0.f, 0.f};
          mma_tf32(d, ax.l, bx.l, az.l, bz.l, yx.h, yz.h);
          mma_tf32(d, ay.l, by.l, aw.l, bw.l, yy.h, yw.h);
          mma_tf32(d, ax.h, bx.h, az.h, bz.h, yx.l, yz.l);
          mma_tf32(d, ay.h, by.h, aw.h, bw.h, yy.l, yw.l);
          mma_tf32(d, ax.h, bx.h, az.h, bz.h, yx.h, yz.h);
          mma_tf32(d, ay.h, by.h, aw.h, bw.h, yy.h, yw.h);
#pragma unroll
          for (int q = 0; q < 4; ++q) w[j][q] += d[q];
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      *reinterpret_cast<float2*>(part + nq * kPW + 8 * j + 2 * kq) = make_float2(w[j][0], w[j][1]);
      *reinterpret_cast<float2*>(part + (nq + 8) * kPW + 8 * j + 2 * kq) = make_float2(w[j][2], w[j][3]);
    }
    team_sync(team);
    {
      // 16 threads per column (half a warp): W, then Z = T^T W (entry i from rows l <= i)
      const int col = tt >> 4, i2 = 2 * (tt & 15);
      const float* src = Pt + team * 8 * (kGC * kPW) + col * kPW + i2;
      float2 s = make_float2(0.f, 0.f);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float2 v = *reinterpret_cast<const float2*>(src + q * (kGC * kPW));
        s.x += v.x;
        s.y += v.y;
      }
      *reinterpret_cast<float2*>(Ws + col * kPW + i2) = s;
      __syncwarp();
      float z0 = 0.f, z1 = 0.f;
#pragma unroll
      for (int l = 0; l < kNb; l += 4) {
        const float4 wv = *reinterpret_cast<const float4*>(Ws + col * kPW + l);
        const float2 t0 = *reinterpret_cast<const float2*>(Tm + l * kNb + i2);
        const float2 t1 = *reinterpret_cast<const float2*>(Tm + (l + 1) * kNb + i2);
        const float2 t2 = *reinterpret_cast<const float2*>(Tm + (l + 2) * kNb + i2);
        const float2 t3 = *reinterpret_cast<const float2*>(Tm + (l + 3) * kNb + i2);
        z0 += t0.x * wv.x + t1.x * wv.y + t2.x * wv.z + t3.x * wv.w;
        z1 += t0.y * wv.x + t1.y * wv.y + t2.y * wv.z + t3.y * wv.w;
      }
      *reinterpret_cast<float2*>(Zt + col * kPW + i2) = make_float2(-z0, -z1);
    }
    team_sync(team);
    if (wr < r) {
      Split z[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        z[j][0] = split_tf32(Zt[nq * kPW + 8 * j + kq]);
        z[j][1] = split_tf32(Zt[(nq + 8) * kPW + 8 * j + kq]);
        z[j][2] = split_tf32(Zt[nq * kPW + 8 * j + kq + 4]);
        z[j][3] = split_tf32(Zt[(nq + 8) * kPW + 8 * j + kq + 4]);
      }
#pragma unroll
      for (int G = 0; G < 8; ++G) {
        const int i = wr + 16 * G;
        float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 u = *reinterpret_cast<const float2*>(Y + ypos(8 * j + kq, i + 2 * nq));
          const float2 v = *reinterpret_cast<const float2*>(Y + ypos(8 * j + kq + 4, i + 2 * nq));
          const Split ux = split_tf32(u.x), uy = split_tf32(u.y), vx = split_tf32(v.x), vy = split_tf32(v.y);
          mma_tf32(d0, z[j][0].l, z[j][1].l, z[j][2].l, z[j][3].l, ux.h, vx.h);
          mma_tf32(d1, z[j][0].l, z[j][1].l, z[j][2].l, z[j][3].l, uy.h, vy.h);
          mma_tf32(d0, z[j][0].h, z[j][1].h, z[j][2].h, z[j][3].h, ux.l, vx.l);
          mma_tf32(d1, z[j][0].h, z[j][1].h, z[j][2].h, z[j][3].h, uy.l, vy.l);
          mma_tf32(d0, z[j][0].h, z[j][1].h, z[j][2].h, z[j][3].h, ux.h, vx.h);
          mma_tf32(d1, z[j][0].h, z[j][1].h, z[j][2].h, z[j][3].h, uy.h, vy.h);
        }
        // rows i + 4 kq, + 1, + 2, + 3 of column nq, then of column nq + 8
        ca[G].x += d0[0]; ca[G].z += d0[1]; cb[G].x += d0[2]; cb[G].z += d0[3];
        ca[G].y += d1[0]; ca[G].w += d1[1]; cb[G].y += d1[2]; cb[G].w += d1[3];
        // the tile's top kmax rows up (the next level, or R_S), the others down (the next panel)
        const int row = i + 4 * kq;
        if (row < r) {
          float* dst;
          int64_t ldd_;
          if (row < kNb) {
            dst = up + (int64_t)(jc + nq) * ldu + tile * kNb + row;
            ldd_ = ldu;
          } else {
            dst = down + (int64_t)(jc + nq) * ldd + down0 + tile * (kTR - kNb) + (row - kNb);
            ldd_ = ldd;
          }
          *reinterpret_cast<float4*>(dst) = ca[G];
          *reinterpret_cast<float4*>(dst + 8 * ldd_) = cb[G];
        }
      }
    }
  }
}

// ---- the tiles' Q^T applied to a right-hand side: y -= Y z, z = T^T (Y^T y) ----
//
// One CTA per tile, thread t owns rows 4 t .. 4 t + 3 and keeps its 32 x 4 reflector entries in
// registers between the two products, so the reflectors are read once, all loads in flight.  z comes
// from G and tau, z_k = tau_k (w_k - sum_{j<k} G[j][k] z_j) with the sum in the order in which row k
// then subtracts Y[k][j] z_j: a column that is zero but for its damping row has a reflector that
// swaps the pivot row out (tau = 1, G[j][k] = Y[k][j]), and row k of the result is then exactly 0,
// as when the reflectors are applied one by one.
constexpr int kQT = kTR / 4;

__global__ void __launch_bounds__(kQT, 1)
tsqr_panel_qt_kernel(const float* X, int64_t ld, int64_t M, const float* Gin, const float* rhs, float* rhs_next,
                     float* rhs_down, int64_t down0) {
  dev::chain_wait();
  __shared__ float ws[kQT / 32][kNb];
  __shared__ float zs[kNb];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t tile = blockIdx.x;
  const int64_t r0 = tile * kTR;
  const int r = (int)(M - r0 < (int64_t)kTR ? M - r0 : (int64_t)kTR);   // a multiple of 4
  const int kmax = r < kNb ? r : kNb;
  const int i = 4 * tid;
  const bool have = i < r;
  float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 v[kNb];
#pragma unroll
  for (int c = 0; c < kNb; ++c) {
    v[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (have && c < kmax) v[c] = *reinterpret_cast<const float4*>(X + (int64_t)c * ld + r0 + i);
  }
  if (have) y = *reinterpret_cast<const float4*>(rhs + r0 + i);
  if (i < kNb) {
#pragma unroll
    for (int c = 0; c < kNb; ++c) {
      const float one = c < kmax ? 1.f : 0.f;
      v[c].x = i > c ? v[c].x : (i == c ? one : 0.f);
      v[c].y = i + 1 > c ? v[c].y : (i + 1 == c ? one : 0.f);
      v[c].z = i + 2 > c ? v[c].z : (i + 2 == c ? one : 0.f);
      v[c].w = i + 3 > c ? v[c].w : (i + 3 == c ? one : 0.f);
    }
  }
  float p[kNb];
#pragma unroll
  for (int c = 0; c < kNb; ++c) p[c] = v[c].x * y.x + v[c].y * y.y + v[c].z * y.z + v[c].w * y.w;
  ws[warp][lane] = transpose_reduce(p, lane);
  __syncthreads();
  if (warp == 0) {
    float w = 0.f;
#pragma unroll
    for (int q = 0; q < kQT / 32; ++q) w += ws[q][lane];
    const float* G = Gin + tile * (kNb * kNb);
    float gc[kNb];   // column `lane` of G above the diagonal
#pragma unroll
    for (int j = 0; j < kNb; ++j) gc[j] = j < lane ? G[j * kNb + lane] : 0.f;
    const float tau = G[lane * kNb + lane];
    float z = 0.f;
#pragma unroll
    for (int j = 0; j < kNb; ++j) {
      if (lane == j) z = tau * w;
      const float zj = __shfl_sync(0xffffffffu, z, j);
      if (j < lane) w = __fmaf_rn(-gc[j], zj, w);
    }
    zs[lane] = z;
  }
  __syncthreads();
  if (!have) return;
#pragma unroll
  for (int c = 0; c < kNb; ++c) {
    const float z = -zs[c];
    y.x = __fmaf_rn(v[c].x, z, y.x);
    y.y = __fmaf_rn(v[c].y, z, y.y);
    y.z = __fmaf_rn(v[c].z, z, y.z);
    y.w = __fmaf_rn(v[c].w, z, y.w);
  }
  if (i < kNb) *reinterpret_cast<float4*>(rhs_next + tile * kNb + i) = y;
  else if (rhs_down) *reinterpret_cast<float4*>(rhs_down + down0 + tile * (kTR - kNb) + (i - kNb)) = y;
}

}  // namespace

// Alignment that every level matrix of a panel has by construction (composed_layout).
static bool panel_aligned(const void* p, int64_t ld, int64_t M) {
  return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 3) == 0 && (M & 3) == 0;
}

qrkit_status tsqr_panel_tile(qrkit_ctx* ctx, float* X, int64_t ld, int64_t M, float* Xn, int64_t ldn, int64_t tiles,
                             float* Tout, float* Gout) {
  if (!panel_aligned(X, ld, M) || !panel_aligned(Xn, ldn, 0))
    return fail(ctx, QRKIT_EINVAL, "column-panel TSQR: unaligned level matrix");
  const unsigned g = (unsigned)tiles;
  auto run = [&](auto k, size_t smem) -> cudaError_t {
    if (smem > 48 * 1024) {
      const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    chain_launch(ctx->stream, g, kPT, smem, k, X, ld, M, Xn, ldn, Tout, Gout, ctx->d_status);
    return cudaSuccess;
  };
  if (M <= 256) QRKIT_CUDA_TRY(ctx, run(tsqr_panel_tile_kernel<2>, panel_tile_smem<2>()));
  else if (M <= 512) QRKIT_CUDA_TRY(ctx, run(tsqr_panel_tile_kernel<4>, panel_tile_smem<4>()));
  else QRKIT_CUDA_TRY(ctx, run(tsqr_panel_tile_kernel<8>, panel_tile_smem<8>()));
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}

qrkit_status tsqr_panel_apply(qrkit_ctx* ctx, const float* X, int64_t ld, int64_t M, const float* T, int n, float* up,
                              int64_t ldu, float* down, int64_t ldd, int64_t down0, int64_t tiles) {
  if (n <= 0 || tiles <= 0) return QRKIT_OK;
  if (!panel_aligned(X, ld, M) || !panel_aligned(up, ldu, 0) || !panel_aligned(down, ldd, down0) || n % kNb != 0)
    return fail(ctx, QRKIT_EINVAL, "column-panel TSQR: unaligned level matrix or panel shape");
  const size_t smem = panel_apply_smem();
  if (smem > ctx->max_smem_optin)
    return fail(ctx, QRKIT_EUNSUPPORTED, "not enough shared memory for the column-panel TSQR kernel");
  if (ctx->smem_attr[15] < smem) {
    QRKIT_CUDA_TRY(ctx, cudaFuncSetAttribute(tsqr_panel_apply_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    ctx->smem_attr[15] = smem;
  }
  // Column ranges: one CTA per SM at a time, so the split that takes the least by waves x (columns of a
  // range + 16, the cost of staging a tile's reflectors in columns).
  int chunk = n;
  int64_t best = INT64_MAX;
  for (int parts = 1; parts <= n / kNb; ++parts) {
    const int ch = (n / kNb + parts - 1) / parts * kNb;
    const int64_t ctas = tiles * ((n + ch - 1) / ch);
    const int64_t cost = (ctas + ctx->num_sms - 1) / ctx->num_sms * (ch + 16);
    if (cost < best) {
      best = cost;
      chunk = ch;
    }
  }
  const dim3 grid((unsigned)tiles, (unsigned)((n + chunk - 1) / chunk));
  chain_launch(ctx->stream, grid, kAT, smem, tsqr_panel_apply_kernel, X, ld, M, T, n, chunk, up, ldu, down, ldd,
               down0);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}

qrkit_status tsqr_panel_qt(qrkit_ctx* ctx, const float* X, int64_t ld, int64_t M, const float* G, const float* rhs,
                           float* rhs_next, float* rhs_down, int64_t down0, int64_t tiles) {
  if (!panel_aligned(X, ld, M) || !panel_aligned(rhs, 0, 0) || !panel_aligned(rhs_next, 0, 0) ||
      !panel_aligned(rhs_down, 0, down0))
    return fail(ctx, QRKIT_EINVAL, "column-panel TSQR: unaligned right-hand side");
  chain_launch(ctx->stream, (unsigned)tiles, kQT, 0, tsqr_panel_qt_kernel, X, ld, M, G, rhs, rhs_next, rhs_down,
               down0);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}

}  // namespace qrkit
