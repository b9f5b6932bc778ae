// Levenberg-Marquardt iterations on the device (Sec. 2; "Backtrack LM" of Sec. 5.2): every
// iteration factors P_r [J; lambda^(1/2) D] once by the composed QR and takes or rejects the
// step by the gain ratio, with Nielsen's damping update.
//
// Model: 2-D points on an open uniform cubic B-spline, one latent parameter t_i per point and
// the control points shared (the block-angular shape of the paper's surface-fitting problems,
// Sec. 6.2 / Fig. 5a): J = [blkdiag(2x1 blocks) | S], each point's two rows touching 8
// consecutive shared columns (a window, Sec. 4.2 + Sec. 4.4).  Several independent problems
// are solved together: their shared columns are separate segments of S, every problem has
// its own lambda, nu and acceptance.
//
//   x = [t of all points | control points of problem 0 (x0, y0, x1, y1, ..), problem 1, ..]
//   seg = clamp(floor(t), 0, Kc - 4), u = t - seg, curve(t) = sum_q B_q(u) P_{seg+q}
//   f_i = curve(t_i) - data_i, cost = 1/2 ||f||^2, b = -f
//   D = column norms of J (zero -> 1); the damping enters as E = lambda_k^(1/2) D per column
//   pred = 1/2 p^T (lambda D^2 p + J^T b) = 1/2 (sum_j E_j^2 p_j^2 + (J p)^T b)
//   rho = (cost(x) - cost(x + p)) / pred (-1 when pred <= 0)
//   Nielsen: rho > 0 -> accept, lambda *= max(1/3, 1 - (2 rho - 1)^3), nu = 2;
//            else lambda *= nu, nu *= 2
// x, the data, residuals and all costs are double; J, S and b are rounded once to the
// context's precision for the factorization.  The state of every problem stays on the device
// between the kernels of an iteration, so an iteration is a fixed sequence of launches and
// can be captured into a CUDA graph (qrkit_lm_run).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <string>
#include <vector>

#include "chain.cuh"
#include "device_util.cuh"
#include "internal.h"
#include "mlp_policy.cuh"
#include "roots.cuh"

namespace qrkit {

constexpr int kTilePts = 256;   // points per reduction tile (tiles never cross problems)

struct LMTables {
  int64_t B = 0, NP = 0, s = 0, N = 0, num_tiles = 0;
  const int64_t* p0 = nullptr;         // B + 1: first point of problem k
  const int64_t* c0 = nullptr;         // B + 1: first shared column of problem k (within S)
  const int64_t* tile_p0 = nullptr;    // num_tiles + 1
  const int32_t* tile_prob = nullptr;  // num_tiles
  const int64_t* prob_tile0 = nullptr; // B + 1
  const int32_t* col_prob = nullptr;   // N: problem of each column
};

struct LM {
  LMTables t;
  std::vector<int64_t> h_p0, h_c0, h_tile_p0, h_prob_tile0;
  DevBuf tabs, tile_prob, col_prob;
  const double* data = nullptr;        // caller's points (device)
  DevBuf J, S, b, p, start, d2, E, coef, tile_cost, tile_new, tile_pred, state, ndone;
  DevBuf hist, feat;                   // per problem: step history (12) and policy features (16)
  bool policy = false;                 // damping from the MLP after accepted steps
  bool prepared = false;
  cudaGraphExec_t graph = nullptr;
  int graph_refine = -1;
  int64_t graph_launches = 0;          // kernels in one captured iteration
  double graph_ftol = 0.0;
  const double* graph_x = nullptr;
};

void release_lm(LM*& lm) {
  if (!lm) return;
  if (lm->graph) cudaGraphExecDestroy(lm->graph);
  for (DevBuf* b : {&lm->tabs, &lm->tile_prob, &lm->col_prob, &lm->J, &lm->S, &lm->b, &lm->p, &lm->start,
                    &lm->d2, &lm->E, &lm->coef, &lm->tile_cost, &lm->tile_new, &lm->tile_pred, &lm->state,
                    &lm->ndone, &lm->hist, &lm->feat})
    release(*b);
  delete lm;
  lm = nullptr;
}

namespace {

// The curve on a segment as a cubic in u = t - seg, from its four control points P0 .. P3:
//   c(u) = a0 + u (a1 + u (a2 + u a3)), c'(u) = a1 + u (2 a2 + 3 a3 u),
//   a0 = (P0 + 4 P1 + P2) / 6, a1 = (P2 - P0) / 2, a2 = (P0 - 2 P1 + P2) / 2, a3 = (P3 - P0 + 3 (P1 - P2)) / 6.
// One thread per segment and coordinate once per evaluation, so that a point costs 10 FP64 multiply-adds instead of
// the basis, its derivative and 16 products: the model kernels are bound by the FP64 unit, which a warp's
// instruction holds for 16 cycles here.  kCoef values per segment: a0 a1 a2 a3 2a2 3a3 for x, then for y.
constexpr int kCoef = 12;

template <typename T>
__global__ void cf_coef_kernel(LMTables t, const double* x, const T* p, double* coef) {
  dev::chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // shared column: control point e / 2, coordinate e % 2
  if (e + 6 >= t.s) return;
  // a segment that starts in the last three control points of a problem mixes two problems' and is never used
  const int64_t j = t.NP + e;
  double P[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) P[q] = x[j + 2 * q] + (p ? (double)p[j + 2 * q] : 0.0);
  double* c = coef + (e / 2) * kCoef + (e & 1) * (kCoef / 2);
  const double a2 = 0.5 * (P[0] + P[2]) - P[1], a3 = (P[3] - P[0] + 3.0 * (P[1] - P[2])) * (1.0 / 6.0);
  c[0] = (P[0] + 4.0 * P[1] + P[2]) * (1.0 / 6.0);
  c[1] = 0.5 * (P[2] - P[0]);
  c[2] = a2;
  c[3] = a3;
  c[4] = 2.0 * a2;
  c[5] = 3.0 * a3;
}

// The basis functions at u, v = 1 - u: B_0 = v^3 / 6, B_1 = (u/2 - 1) u^2 + 2/3, and the same mirrored.
__device__ __forceinline__ void bspline_values(double u, double B[4]) {
  const double sixth = 1.0 / 6.0;
  const double v = 1.0 - u, u2 = u * u, v2 = v * v;
  B[0] = v2 * v * sixth;
  B[1] = fma(fma(0.5, u, -1.0), u2, 4.0 * sixth);
  B[2] = fma(fma(0.5, v, -1.0), v2, 4.0 * sixth);
  B[3] = u2 * u * sixth;
}

// Segment of parameter t and u = t - segment.
__device__ __forceinline__ int segment_of(double t, int64_t Kc, double& u) {
  const int f = max(0, min(__double2int_rd(t), (int)(Kc - 4)));   // saturates; NaN becomes a negative number or 0
  u = t - (double)f;
  return f;
}

// Sum over the CTA of kTilePts threads, in thread 0: through shared memory, so that the FP64 additions are those of
// one warp.
__device__ __forceinline__ double tile_sum(double v, double* buf) {
  buf[threadIdx.x] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
#pragma unroll
    for (int q = 0; q < kTilePts / 32; ++q) s += buf[threadIdx.x + 32 * q];
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
  }
  return s;
}

// Residual, Jacobian blocks, windows, b = -f and the cost per tile.
template <typename T>
__global__ void __launch_bounds__(kTilePts)
cf_eval_kernel(LMTables t, const double* x, const double* data, const double* coef, T* J, T* S, T* b, int32_t* start,
               double* tile_cost) {
  dev::chain_wait();
  __shared__ double red[kTilePts];
  const int64_t tile = blockIdx.x;
  const int64_t i = t.tile_p0[tile] + threadIdx.x;
  double fsq = 0.0;
  if (i < t.tile_p0[tile + 1]) {
    const int k = t.tile_prob[tile];
    const int64_t c0 = t.c0[k], Kc = (t.c0[k + 1] - c0) / 2;
    double u;
    const int seg = segment_of(x[i], Kc, u);
    const double2* c = reinterpret_cast<const double2*>(coef + (c0 / 2 + seg) * kCoef);
    const double2 x01 = c[0], x23 = c[1], xd = c[2], y01 = c[3], y23 = c[4], yd = c[5];
    const double fx = fma(fma(fma(x23.y, u, x23.x), u, x01.y), u, x01.x) - data[2 * i];
    const double fy = fma(fma(fma(y23.y, u, y23.x), u, y01.y), u, y01.x) - data[2 * i + 1];
    fsq = fma(fx, fx, fy * fy);
    J[2 * i] = (T)fma(fma(xd.y, u, xd.x), u, x01.y);
    J[2 * i + 1] = (T)fma(fma(yd.y, u, yd.x), u, y01.y);
    b[2 * i] = (T)(-fx);
    b[2 * i + 1] = (T)(-fy);
    start[i] = (int32_t)(c0 + 2 * seg);
    double B[4];
    bspline_values(u, B);
    T* Si = S + 16 * i;   // 2 x 8, column-major: (B_q, 0) for column 2 q, (0, B_q) for column 2 q + 1
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const T v = (T)B[q];
      if constexpr (sizeof(T) == 4) {
        reinterpret_cast<float4*>(Si)[q] = make_float4(v, 0.f, 0.f, v);
      } else {
        reinterpret_cast<double2*>(Si)[2 * q] = make_double2(v, 0.0);
        reinterpret_cast<double2*>(Si)[2 * q + 1] = make_double2(0.0, v);
      }
    }
  }
  const double s = tile_sum(fsq, red);
  if (threadIdx.x == 0) tile_cost[tile] = s;
}

// E_j = lambda_k^(1/2) D_j with D_j = ||column j of J|| (zero -> 1): a tile of points per CTA, then the shared
// columns (squared norms d2) 256 at a time.
template <typename T>
__global__ void __launch_bounds__(kTilePts) lm_damp_kernel(LMTables t, const T* J, const double* d2,
                                                           const qrkit_lm_state* st, double* E) {
  dev::chain_wait();
  __shared__ double root;
  if (blockIdx.x < t.num_tiles) {
    const int64_t tile = blockIdx.x, i = t.tile_p0[tile] + threadIdx.x;
    if (threadIdx.x == 0) root = sqrt(st[t.tile_prob[tile]].lambda);
    __syncthreads();
    if (i >= t.tile_p0[tile + 1]) return;
    const T jx = J[2 * i], jy = J[2 * i + 1];
    double d;
    if constexpr (sizeof(T) == 4) d = dev::norm_of_two(jx, jy);
    else d = sqrt(jx * jx + jy * jy);
    E[i] = root * (d == 0.0 ? 1.0 : d);
    return;
  }
  const int64_t c = (blockIdx.x - t.num_tiles) * (int64_t)kTilePts + threadIdx.x;
  if (c >= t.s) return;
  const double d = sqrt(d2[c]);
  E[t.NP + c] = sqrt(st[t.col_prob[t.NP + c]].lambda) * (d == 0.0 ? 1.0 : d);
}

// f = curve(t) - data per point (two values), double.
__global__ void cf_residual_kernel(LMTables t, const double* x, const double* data, double* f) {
  dev::chain_wait();
  const int64_t tile = blockIdx.x;
  const int64_t i = t.tile_p0[tile] + threadIdx.x;
  if (i >= t.tile_p0[tile + 1]) return;
  const int k = t.tile_prob[tile];
  const int64_t Kc = (t.c0[k + 1] - t.c0[k]) / 2;
  double u, Bv[4];
  const int seg = segment_of(x[i], Kc, u);
  bspline_values(u, Bv);
  const double* P = x + t.NP + t.c0[k] + 2 * seg;
  double cx = 0, cy = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    cx += Bv[q] * P[2 * q];
    cy += Bv[q] * P[2 * q + 1];
  }
  f[2 * i] = cx - data[2 * i];
  f[2 * i + 1] = cy - data[2 * i + 1];
}

// Cost at x + p and the row part of the predicted decrease, (J p)^T b + E_t^2 p_t^2, per tile.
template <typename T>
__global__ void __launch_bounds__(kTilePts)
cf_trial_kernel(LMTables t, const double* x, const double* data, const double* coef, const T* J, const T* S, const T* b,
                const T* p, const double* E, const int32_t* start, double* tile_new, double* tile_pred) {
  dev::chain_wait();
  __shared__ double red[2][kTilePts];
  const int64_t tile = blockIdx.x;
  const int64_t i = t.tile_p0[tile] + threadIdx.x;
  double fsq = 0.0, pr = 0.0;
  if (i < t.tile_p0[tile + 1]) {
    const int k = t.tile_prob[tile];
    const int64_t Kc = (t.c0[k + 1] - t.c0[k]) / 2;
    const T pt = p[i];
    double u;
    const int seg = segment_of(x[i] + (double)pt, Kc, u);
    const double2* c = reinterpret_cast<const double2*>(coef + (t.c0[k] / 2 + seg) * kCoef);   // of x + p
    const double2 x01 = c[0], x23 = c[1], y01 = c[3], y23 = c[4];
    const double fx = fma(fma(fma(x23.y, u, x23.x), u, x01.y), u, x01.x) - data[2 * i];
    const double fy = fma(fma(fma(y23.y, u, y23.x), u, y01.y), u, y01.x) - data[2 * i + 1];
    fsq = fma(fx, fx, fy * fy);
    // (J p) at the linearisation point, with the system's own J, S and b; in the context
    // precision (a relative error of the order of its rounding in the predicted decrease moves
    // the gain ratio by as little, far below what the damping rule resolves)
    T jx = J[2 * i] * pt, jy = J[2 * i + 1] * pt;
    const T* Si = S + 16 * i;
    const T* pS = p + t.NP + start[i];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      jx += Si[2 * c] * pS[c];
      jy += Si[2 * c + 1] * pS[c];
    }
    const T e = (T)E[i];
    pr = (double)(jx * b[2 * i] + jy * b[2 * i + 1] + e * e * pt * pt);
  }
  const double s1 = tile_sum(fsq, red[0]);
  const double s2 = tile_sum(pr, red[1]);
  if (threadIdx.x == 0) {
    tile_new[tile] = s1;
    tile_pred[tile] = s2;
  }
}

constexpr int kUpdateThreads = 256;
constexpr int kHist = 12;   // rho, accepted, log cost ratio of the last 4 steps

__device__ __forceinline__ float clampf(float v, float lo, float hi) { return fminf(fmaxf(v, lo), hi); }

// One CTA per problem (a warp, or eight for few problems): costs, predicted decrease, gain ratio, then on its first
// warp the damping update:
// Nielsen's rule, or after an accepted step (when the policy is on) lambda * multiplier of the
// MLP's class for the features of the step history; stop rule.
template <typename T>
__global__ void lm_update_kernel(LMTables t, const double* tile_cost, const double* tile_new,
                                 const double* tile_pred, const double* E, const T* p, qrkit_lm_state* st,
                                 double ftol, int* ndone, MlpDev w, float* hist, float* feat) {
  dev::chain_wait();
  __shared__ double part[3][kUpdateThreads / 32];
  const int64_t k = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double c = 0, cn = 0, pr = 0;
  for (int64_t q = t.prob_tile0[k] + threadIdx.x; q < t.prob_tile0[k + 1]; q += blockDim.x) {
    c += tile_cost[q];
    cn += tile_new[q];
    pr += tile_pred[q];
  }
  for (int64_t j = t.NP + t.c0[k] + threadIdx.x; j < t.NP + t.c0[k + 1]; j += blockDim.x) {
    const double pj = (double)p[j];
    pr += E[j] * E[j] * pj * pj;
  }
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    c += __shfl_xor_sync(0xffffffffu, c, d);
    cn += __shfl_xor_sync(0xffffffffu, cn, d);
    pr += __shfl_xor_sync(0xffffffffu, pr, d);
  }
  if (nw > 1) {
    if (lane == 0) {
      part[0][warp] = c;
      part[1][warp] = cn;
      part[2][warp] = pr;
    }
    __syncthreads();
    if (warp > 0) return;
    c = cn = pr = 0.0;
    for (int q = 0; q < nw; ++q) {
      c += part[0][q];
      cn += part[1][q];
      pr += part[2][q];
    }
  }
  qrkit_lm_state s = st[k];
  if (s.done) {
    if (lane == 0) {
      s.accepted = 0;
      st[k] = s;
      atomicAdd(ndone, 1);
    }
    return;
  }
  const double cost = 0.5 * c, cost_new = 0.5 * cn, pred = 0.5 * pr;
  const double rho = pred > 0.0 ? (cost - cost_new) / pred : -1.0;
  const bool acc = rho > 0.0;
  // step history and features (every lane computes the same values)
  float* hk = hist + k * kHist;
  float h[kHist];
#pragma unroll
  for (int q = 0; q < kHist; ++q) h[q] = s.iteration == 0 ? 0.f : hk[q];
  const float ratio = cost > 0.0 ? (float)log10(fmax(cost_new / cost, 1e-30)) : 0.f;
  const float pratio = cost > 0.0 ? (float)log10(fmax(pred / cost, 1e-30)) : -16.f;
#pragma unroll
  for (int q = 3; q >= 1; --q) {
    h[q] = h[q - 1];
    h[4 + q] = h[4 + q - 1];
    h[8 + q] = h[8 + q - 1];
  }
  h[0] = clampf((float)rho, -1.f, 2.f);
  h[4] = acc ? 1.f : 0.f;
  h[8] = clampf(ratio, -8.f, 1.f) / 8.f;
  float f[kMlpF];
  f[0] = (float)log10(s.lambda) / 4.f;
  f[1] = (float)log10((double)(s.iteration + 1)) / 2.f;
#pragma unroll
  for (int q = 0; q < kHist; ++q) f[2 + q] = h[q];
  f[14] = clampf(pratio, -16.f, 0.f) / 16.f;
  f[15] = 1.f;
  __syncwarp();
  if (lane < kHist) hk[lane] = h[lane];
  if (lane < kMlpF) feat[k * kMlpF + lane] = f[lane];
  int cls = -1;
  if (acc && w.theta) cls = mlp_policy_warp(w, f, lane);
  if (lane != 0) return;
  s.cost = cost;
  s.cost_new = cost_new;
  s.pred = pred;
  s.rho = rho;
  if (acc) {
    if (cls >= 0) {
      s.lambda *= mlp_multiplier(cls);
    } else {
      const double a = 2.0 * rho - 1.0;
      s.lambda *= fmax(1.0 / 3.0, 1.0 - a * a * a);
    }
    s.nu = 2.0;
    s.accepted = 1;
    if (ftol >= 0.0 && cost - cost_new <= ftol * cost) s.done = 1;
  } else {
    s.lambda *= s.nu;
    s.nu *= 2.0;
    s.accepted = 0;
  }
  if (s.lambda > 1e16) s.done = 1;
  if (s.lambda < 1e-30) s.lambda = 1e-30;
  s.iteration += 1;
  st[k] = s;
  if (s.done) atomicAdd(ndone, 1);
}

template <typename T>
__global__ void lm_accept_kernel(LMTables t, const T* p, double* x, const qrkit_lm_state* st) {
  dev::chain_wait();
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= t.N) return;
  if (st[t.col_prob[j]].accepted) x[j] += (double)p[j];
}

inline unsigned nblk(int64_t n, int th) { return (unsigned)((n + th - 1) / th); }

#define LM_LAUNCH(ctx, ...)                         \
  do {                                              \
    __VA_ARGS__;                                    \
    (ctx)->launches += 1;                           \
    QRKIT_CUDA_TRY(ctx, cudaGetLastError());        \
  } while (0)

// One LM iteration for every problem (all work on ctx->stream; no host synchronisation).
template <typename T>
qrkit_status lm_iteration(qrkit_ctx* ctx, double* x, int refine_steps, double ftol) {
  LM& L = *ctx->lm;
  const LMTables& t = L.t;
  cudaStream_t st = ctx->stream;
  qrkit_lm_state* S = (qrkit_lm_state*)L.state.ptr;
  T* J = (T*)L.J.ptr;
  T* Sv = (T*)L.S.ptr;
  T* b = (T*)L.b.ptr;
  T* p = (T*)L.p.ptr;
  double* d2 = (double*)L.d2.ptr;
  double* E = (double*)L.E.ptr;
  double* coef = (double*)L.coef.ptr;
  int32_t* start = (int32_t*)ctx->plan.d_start.ptr;   // the model's starts lie in their segments
  QRKIT_CUDA_TRY(ctx, cudaMemsetAsync(L.ndone.ptr, 0, sizeof(int), st));
  LM_LAUNCH(ctx, chain_launch(st, nblk(t.s, 128), 128, 0, cf_coef_kernel<T>, t, x, (const T*)nullptr, coef));
  LM_LAUNCH(ctx, chain_launch(st, (unsigned)t.num_tiles, kTilePts, 0, cf_eval_kernel<T>, t, x, L.data, coef, J, Sv, b,
                              start, (double*)L.tile_cost.ptr));
  bool sorted = false;
  qrkit_status rc = composed_sort_blocks(ctx, &sorted);
  if (rc != QRKIT_OK) return rc;
  if (!sorted) return fail(ctx, QRKIT_ESTATE, "the LM plan has no block sort");
  if ((rc = composed_window_sums(ctx, Sv, d2)) != QRKIT_OK) return rc;
  LM_LAUNCH(ctx, chain_launch(st, (unsigned)(t.num_tiles + (t.s + kTilePts - 1) / kTilePts), kTilePts, 0,
                              lm_damp_kernel<T>, t, J, d2, S, E));
  if ((rc = composed_factor_scaled(ctx, J, Sv, E, true)) != QRKIT_OK) return rc;
  if ((rc = composed_solve(ctx, true, J, Sv, b, p, refine_steps)) != QRKIT_OK) return rc;
  LM_LAUNCH(ctx, chain_launch(st, nblk(t.s, 128), 128, 0, cf_coef_kernel<T>, t, x, p, coef));
  LM_LAUNCH(ctx, chain_launch(st, (unsigned)t.num_tiles, kTilePts, 0, cf_trial_kernel<T>, t, x, L.data, coef, J, Sv,
                              b, p, E, start, (double*)L.tile_new.ptr, (double*)L.tile_pred.ptr));
  MlpDev w{};
  if (L.policy && ctx->mlp) {
    w.theta = (const float*)ctx->mlp->theta.ptr;
    w.wbf = (const __nv_bfloat16*)ctx->mlp->wbf.ptr;
  }
  LM_LAUNCH(ctx, chain_launch(st, (unsigned)t.B, t.B >= 2 * ctx->num_sms ? 32 : kUpdateThreads, 0,
                              lm_update_kernel<T>, t, (const double*)L.tile_cost.ptr, (const double*)L.tile_new.ptr,
                              (const double*)L.tile_pred.ptr, E, p, S, ftol, (int*)L.ndone.ptr, w, (float*)L.hist.ptr,
                              (float*)L.feat.ptr));
  LM_LAUNCH(ctx, chain_launch(st, nblk(t.N, 256), 256, 0, lm_accept_kernel<T>, t, p, x, S));
  return QRKIT_OK;
}

qrkit_status iterate(qrkit_ctx* ctx, double* x, int refine_steps, double ftol) {
  if (ctx->precision == QRKIT_FP64) return lm_iteration<double>(ctx, x, refine_steps, ftol);
  return lm_iteration<float>(ctx, x, refine_steps, ftol);
}

// Allocations and uploads of the composed factor happen here, outside any stream capture.
qrkit_status lm_prepare(qrkit_ctx* ctx) {
  LM& L = *ctx->lm;
  if (L.prepared) return QRKIT_OK;
  Composed& C = ctx->comp;
  C.damp = true;
  C.lam = 1.0;
  C.lam_half = 1.0;
  qrkit_status rc = composed_layout(ctx, elem_size(ctx));
  if (rc != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.D, (size_t)L.t.N * sizeof(double), "D")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, C.sq, (size_t)L.t.N * sizeof(double), "column sums")) != QRKIT_OK) return rc;
  L.prepared = true;
  return QRKIT_OK;
}

qrkit_status check_ready(qrkit_ctx* ctx, double* x, qrkit_lm_state* states, int refine_steps) {
  if (!ctx->lm) return fail(ctx, QRKIT_ESTATE, "no LM model planned (qrkit_lm_plan)");
  if (!x || !states) return fail(ctx, QRKIT_EINVAL, "x and states are required");
  if (refine_steps < 0 || refine_steps > 8) return fail(ctx, QRKIT_EINVAL, "refine_steps must be in [0, 8]");
  for (int64_t k = 0; k < ctx->lm->t.B; ++k)
    if (!(states[k].lambda > 0.0) || !(states[k].nu >= 1.0))
      return fail(ctx, QRKIT_EINVAL, "problem " + std::to_string(k) + ": lambda must be > 0 and nu >= 1");
  return QRKIT_OK;
}

qrkit_status read_status(qrkit_ctx* ctx) {
  QRKIT_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
  int h = 0;
  QRKIT_CUDA_TRY(ctx, cudaMemcpy(&h, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost));
  if (h != 0) {
    QRKIT_CUDA_TRY(ctx, cudaMemset(ctx->d_status, 0, sizeof(int)));
    return fail(ctx, (qrkit_status)h, std::string("device reported ") + qrkit_status_string(h));
  }
  return QRKIT_OK;
}

}  // namespace
}  // namespace qrkit

using namespace qrkit;

extern "C" {

qrkit_status qrkit_lm_plan(qrkit_ctx* ctx, const qrkit_lm_problem* pr) {
  if (!ctx) return QRKIT_EINVAL;
  if (!pr) return fail(ctx, QRKIT_EINVAL, "null problem");
  if (pr->model != QRKIT_MODEL_CURVEFIT) return fail(ctx, QRKIT_EUNSUPPORTED, "unknown model");
  if (pr->num_problems < 1 || !pr->num_points || !pr->control_points || !pr->data)
    return fail(ctx, QRKIT_EINVAL, "num_problems >= 1, num_points, control_points and data are required");
  const int64_t B = pr->num_problems;
  std::vector<int64_t> p0(B + 1, 0), c0(B + 1, 0);
  for (int64_t k = 0; k < B; ++k) {
    if (pr->num_points[k] < 1) return fail(ctx, QRKIT_EINVAL, "problem " + std::to_string(k) + " has no points");
    if (pr->control_points[k] < 4)
      return fail(ctx, QRKIT_EINVAL, "problem " + std::to_string(k) + " needs at least 4 control points");
    p0[k + 1] = p0[k] + pr->num_points[k];
    c0[k + 1] = c0[k] + 2 * (int64_t)pr->control_points[k];
  }
  const int64_t NP = p0[B], s = c0[B];
  if (NP >= ((int64_t)1 << 31) || s >= ((int64_t)1 << 31))
    return fail(ctx, QRKIT_EUNSUPPORTED, "more than 2^31 points or shared columns");
  // block-angular structure: 2x1 blocks, windows of 8 shared columns, one segment per problem
  std::vector<uint8_t> n(NP, 2), m(NP, 1);
  std::vector<int32_t> ws(NP);
  std::vector<int64_t> seg_cols(B), seg_blocks(B);
  for (int64_t k = 0; k < B; ++k) {
    seg_cols[k] = c0[k + 1] - c0[k];
    seg_blocks[k] = p0[k + 1] - p0[k];
    for (int64_t i = p0[k]; i < p0[k + 1]; ++i) ws[i] = (int32_t)c0[k];
  }
  qrkit_structure st{};
  st.kind = QRKIT_STRUCT_BLOCKS;
  st.num_blocks = NP;
  st.block_rows = n.data();
  st.block_cols = m.data();
  st.coupled_kind = QRKIT_COUPLED_WINDOW;
  st.shared_cols = s;
  st.window = 8;
  st.window_start = ws.data();
  st.num_segments = B;
  st.segment_cols = seg_cols.data();
  st.segment_blocks = seg_blocks.data();
  qrkit_status rc = qrkit_plan(ctx, &st);   // releases any previous LM state
  if (rc != QRKIT_OK) return rc;
  ctx->lm = new LM();
  LM& L = *ctx->lm;
  L.t.B = B;
  L.t.NP = NP;
  L.t.s = s;
  L.t.N = NP + s;
  L.h_p0 = p0;
  L.h_c0 = c0;
  L.h_tile_p0.clear();
  L.h_prob_tile0.assign(B + 1, 0);
  std::vector<int32_t> tile_prob;
  for (int64_t k = 0; k < B; ++k) {
    L.h_prob_tile0[k] = (int64_t)L.h_tile_p0.size();
    for (int64_t q = p0[k]; q < p0[k + 1]; q += kTilePts) {
      L.h_tile_p0.push_back(q);
      tile_prob.push_back((int32_t)k);
    }
  }
  L.h_prob_tile0[B] = (int64_t)L.h_tile_p0.size();
  L.t.num_tiles = (int64_t)L.h_tile_p0.size();
  L.h_tile_p0.push_back(NP);
  std::vector<int32_t> col_prob(L.t.N);
  for (int64_t k = 0; k < B; ++k) {
    for (int64_t i = p0[k]; i < p0[k + 1]; ++i) col_prob[i] = (int32_t)k;
    for (int64_t c = c0[k]; c < c0[k + 1]; ++c) col_prob[NP + c] = (int32_t)k;
  }
  std::vector<int64_t> tabs;
  for (auto* v : {&p0, &c0, &L.h_tile_p0, &L.h_prob_tile0}) tabs.insert(tabs.end(), v->begin(), v->end());
  const size_t es = elem_size(ctx);
  auto up = [&](DevBuf& d, const void* h, size_t bytes, const char* what) -> qrkit_status {
    qrkit_status r = ensure(ctx, d, bytes, what);
    if (r != QRKIT_OK) return r;
    QRKIT_CUDA_TRY(ctx, cudaMemcpy(d.ptr, h, bytes, cudaMemcpyHostToDevice));
    return QRKIT_OK;
  };
  if ((rc = up(L.tabs, tabs.data(), tabs.size() * sizeof(int64_t), "LM tables")) != QRKIT_OK) return rc;
  if ((rc = up(L.tile_prob, tile_prob.data(), tile_prob.size() * sizeof(int32_t), "LM tiles")) != QRKIT_OK) return rc;
  if ((rc = up(L.col_prob, col_prob.data(), col_prob.size() * sizeof(int32_t), "LM columns")) != QRKIT_OK) return rc;
  const int64_t* tb = (const int64_t*)L.tabs.ptr;
  L.t.p0 = tb;
  L.t.c0 = tb + (B + 1);
  L.t.tile_p0 = tb + 2 * (B + 1);
  L.t.prob_tile0 = tb + 2 * (B + 1) + (L.t.num_tiles + 1);
  L.t.tile_prob = (const int32_t*)L.tile_prob.ptr;
  L.t.col_prob = (const int32_t*)L.col_prob.ptr;
  L.data = pr->data;
  const int64_t N = L.t.N, nt = L.t.num_tiles;
  if ((rc = ensure(ctx, L.J, (size_t)2 * NP * es, "LM J")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.S, (size_t)16 * NP * es, "LM S")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.b, (size_t)2 * NP * es, "LM b")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.p, (size_t)N * es, "LM p")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.start, (size_t)NP * sizeof(int32_t), "LM starts")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.d2, (size_t)s * sizeof(double), "LM norms")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.E, (size_t)N * sizeof(double), "LM damping")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.coef, (size_t)(s / 2) * kCoef * sizeof(double), "LM segments")) != QRKIT_OK) return rc;
  for (DevBuf* d : {&L.tile_cost, &L.tile_new, &L.tile_pred})
    if ((rc = ensure(ctx, *d, (size_t)nt * sizeof(double), "LM partial sums")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.state, (size_t)B * sizeof(qrkit_lm_state), "LM state")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.ndone, sizeof(int), "LM done count")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.hist, (size_t)B * kHist * sizeof(float), "LM history")) != QRKIT_OK) return rc;
  if ((rc = ensure(ctx, L.feat, (size_t)B * kMlpF * sizeof(float), "LM features")) != QRKIT_OK) return rc;
  QRKIT_CUDA_TRY(ctx, cudaMemset(L.hist.ptr, 0, (size_t)B * kHist * sizeof(float)));
  QRKIT_CUDA_TRY(ctx, cudaMemset(L.feat.ptr, 0, (size_t)B * kMlpF * sizeof(float)));
  return QRKIT_OK;
}

qrkit_status qrkit_lm_linearize(qrkit_ctx* ctx, const double* x, void* J, void* S, void* b, int32_t* start) {
  if (!ctx) return QRKIT_EINVAL;
  if (!ctx->lm) return fail(ctx, QRKIT_ESTATE, "no LM model planned (qrkit_lm_plan)");
  if (!x) return fail(ctx, QRKIT_EINVAL, "x is required");
  QRKIT_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  LM& L = *ctx->lm;
  const LMTables& t = L.t;
  cudaStream_t st = ctx->stream;
  const double* coef = (const double*)L.coef.ptr;
  if (ctx->precision == QRKIT_FP64) {
    start_launch(st, nblk(t.s, 128), 128, 0, cf_coef_kernel<double>, t, x, (const double*)nullptr,
                 (double*)L.coef.ptr);
    chain_launch(st, (unsigned)t.num_tiles, kTilePts, 0, cf_eval_kernel<double>, t, x, L.data, coef, (double*)L.J.ptr,
                 (double*)L.S.ptr, (double*)L.b.ptr, (int32_t*)L.start.ptr, (double*)L.tile_cost.ptr);
  } else {
    start_launch(st, nblk(t.s, 128), 128, 0, cf_coef_kernel<float>, t, x, (const float*)nullptr, (double*)L.coef.ptr);
    chain_launch(st, (unsigned)t.num_tiles, kTilePts, 0, cf_eval_kernel<float>, t, x, L.data, coef, (float*)L.J.ptr,
                 (float*)L.S.ptr, (float*)L.b.ptr, (int32_t*)L.start.ptr, (double*)L.tile_cost.ptr);
  }
  ctx->launches += 2;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  const size_t es = elem_size(ctx);
  if (J) QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(J, L.J.ptr, (size_t)2 * t.NP * es, cudaMemcpyDeviceToDevice, st));
  if (S) QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(S, L.S.ptr, (size_t)16 * t.NP * es, cudaMemcpyDeviceToDevice, st));
  if (b) QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(b, L.b.ptr, (size_t)2 * t.NP * es, cudaMemcpyDeviceToDevice, st));
  if (start)
    QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(start, L.start.ptr, (size_t)t.NP * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
  return QRKIT_OK;
}

qrkit_status qrkit_lm_residual(qrkit_ctx* ctx, const double* x, double* f) {
  if (!ctx) return QRKIT_EINVAL;
  if (!ctx->lm) return fail(ctx, QRKIT_ESTATE, "no LM model planned (qrkit_lm_plan)");
  if (!x || !f) return fail(ctx, QRKIT_EINVAL, "x and f are required");
  QRKIT_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  LM& L = *ctx->lm;
  start_launch(ctx->stream, (unsigned)L.t.num_tiles, kTilePts, 0, cf_residual_kernel, L.t, x, L.data, f);
  ctx->launches += 1;
  QRKIT_CUDA_TRY(ctx, cudaGetLastError());
  return QRKIT_OK;
}

qrkit_status qrkit_lm_set_policy(qrkit_ctx* ctx, int use_mlp) {
  if (!ctx) return QRKIT_EINVAL;
  if (!ctx->lm) return fail(ctx, QRKIT_ESTATE, "no LM model planned (qrkit_lm_plan)");
  if (use_mlp && !ctx->mlp) return fail(ctx, QRKIT_ESTATE, "no MLP (qrkit_mlp_init)");
  LM& L = *ctx->lm;
  if (L.policy != (use_mlp != 0) && L.graph) {
    cudaGraphExecDestroy(L.graph);
    L.graph = nullptr;
  }
  L.policy = use_mlp != 0;
  return QRKIT_OK;
}

qrkit_status qrkit_lm_features(qrkit_ctx* ctx, float* features) {
  if (!ctx) return QRKIT_EINVAL;
  if (!ctx->lm) return fail(ctx, QRKIT_ESTATE, "no LM model planned (qrkit_lm_plan)");
  if (!features) return fail(ctx, QRKIT_EINVAL, "features is required");
  LM& L = *ctx->lm;
  QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(features, L.feat.ptr, (size_t)L.t.B * kMlpF * sizeof(float),
                                      cudaMemcpyDeviceToDevice, ctx->stream));
  return QRKIT_OK;
}

qrkit_status qrkit_lm_step(qrkit_ctx* ctx, double* x, qrkit_lm_state* states, int refine_steps) {
  if (!ctx) return QRKIT_EINVAL;
  qrkit_status rc = check_ready(ctx, x, states, refine_steps);
  if (rc != QRKIT_OK) return rc;
  QRKIT_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  if ((rc = lm_prepare(ctx)) != QRKIT_OK) return rc;
  LM& L = *ctx->lm;
  const size_t sb = (size_t)L.t.B * sizeof(qrkit_lm_state);
  QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(L.state.ptr, states, sb, cudaMemcpyHostToDevice, ctx->stream));
  if ((rc = iterate(ctx, x, refine_steps, -1.0)) != QRKIT_OK) return rc;
  ctx->comp_factored = true;
  QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(states, L.state.ptr, sb, cudaMemcpyDeviceToHost, ctx->stream));
  return read_status(ctx);
}

qrkit_status qrkit_lm_run(qrkit_ctx* ctx, double* x, qrkit_lm_state* states, int max_iter, double ftol,
                          int refine_steps, int use_graph) {
  if (!ctx) return QRKIT_EINVAL;
  qrkit_status rc = check_ready(ctx, x, states, refine_steps);
  if (rc != QRKIT_OK) return rc;
  if (max_iter < 0) return fail(ctx, QRKIT_EINVAL, "max_iter must be >= 0");
  if (!(ftol >= 0.0)) return fail(ctx, QRKIT_EINVAL, "ftol must be >= 0");
  QRKIT_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  if ((rc = lm_prepare(ctx)) != QRKIT_OK) return rc;
  LM& L = *ctx->lm;
  cudaStream_t st = ctx->stream;
  const size_t sb = (size_t)L.t.B * sizeof(qrkit_lm_state);
  QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(L.state.ptr, states, sb, cudaMemcpyHostToDevice, st));
  if (use_graph && (!L.graph || L.graph_refine != refine_steps || L.graph_ftol != ftol || L.graph_x != x)) {
    // capture one iteration (kernel arguments are fixed: x must stay the same buffer)
    if (L.graph) {
      cudaGraphExecDestroy(L.graph);
      L.graph = nullptr;
    }
    const int64_t before = ctx->launches;
    QRKIT_CUDA_TRY(ctx, cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
    rc = iterate(ctx, x, refine_steps, ftol);
    cudaGraph_t g = nullptr;
    const cudaError_t e = cudaStreamEndCapture(st, &g);
    if (rc != QRKIT_OK) {
      if (g) cudaGraphDestroy(g);
      return rc;
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaStreamEndCapture");
    const cudaError_t e2 = cudaGraphInstantiate(&L.graph, g, 0);
    cudaGraphDestroy(g);
    if (e2 != cudaSuccess) return cuda_fail(ctx, e2, "cudaGraphInstantiate");
    L.graph_launches = ctx->launches - before;
    ctx->launches = before;
    L.graph_refine = refine_steps;
    L.graph_ftol = ftol;
    L.graph_x = x;
  }
  int done = 0;
  for (int it = 0; it < max_iter; ++it) {
    if (use_graph) {
      QRKIT_CUDA_TRY(ctx, cudaGraphLaunch(L.graph, st));
      ctx->launches += L.graph_launches;
    } else if ((rc = iterate(ctx, x, refine_steps, ftol)) != QRKIT_OK) {
      return rc;
    }
    if ((it + 1) % 8 == 0 || it + 1 == max_iter) {
      QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(&done, L.ndone.ptr, sizeof(int), cudaMemcpyDeviceToHost, st));
      QRKIT_CUDA_TRY(ctx, cudaStreamSynchronize(st));
      if (done >= L.t.B) break;
    }
  }
  ctx->comp_factored = true;
  QRKIT_CUDA_TRY(ctx, cudaMemcpyAsync(states, L.state.ptr, sb, cudaMemcpyDeviceToHost, st));
  return read_status(ctx);
}

}  // extern "C"
