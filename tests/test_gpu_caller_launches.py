"""Calls behind a caller's own kernels launched by programmatic dependent launch: an input written by a kernel that is
still running when the caller's last kernel, which does not wait for it, has ended.  Every call's first launch is
ordered behind both."""
import ctypes
import subprocess

import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cuda_runtime.h>
// Lets the next kernel start, runs for `cycles` clocks, then copies n words.
__global__ void late_copy(unsigned* dst, const unsigned* src, long long n, long long cycles) {
  asm volatile("griddepcontrol.launch_dependents;");
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) {}
  for (long long i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}
__global__ void nothing() {}
extern "C" int late_input(void* dst, const void* src, long long bytes, long long cycles, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  late_copy<<<1, 1024, 0, st>>>((unsigned*)dst, (const unsigned*)src, bytes / 4, cycles);
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = 1;
  c.blockDim = 32;
  c.stream = st;
  c.attrs = &a;
  c.numAttrs = 1;
  return (int)cudaLaunchKernelEx(&c, nothing);
}
"""


@pytest.fixture(scope="module")
def late_input(tmp_path_factory):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import build
    d = tmp_path_factory.mktemp("late")
    (d / "late.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", str(d / "late.so"),
                    str(d / "late.cu")], check=True, capture_output=True)
    fn = ctypes.CDLL(str(d / "late.so")).late_input
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_void_p]

    def run(dst, src, stream):
        assert fn(dst.data_ptr(), src.data_ptr(), dst.numel() * dst.element_size(), 2_000_000, stream.cuda_stream) == 0
    return torch, run


def both(torch, late, ctx, stream, src, call, out):
    """The call's output with its input in place, and with the input written behind the caller's chained kernel."""
    dst = src.clone()
    torch.cuda.synchronize()
    call(dst)
    ctx.sync_status()
    want = out.clone()
    dst.zero_()
    out.zero_()
    torch.cuda.synchronize()
    late(dst, src, stream)
    call(dst)
    ctx.sync_status()
    torch.cuda.synchronize()
    return want, out


def check(torch, late, ctx, stream, src, call, out):
    want, got = both(torch, late, ctx, stream, src, call, out)
    assert want.abs().max() > 0 and torch.equal(got, want)


def test_banded(late_input):
    torch, late = late_input
    from paper_1802_03773_gb300 import Context
    g = np.random.default_rng(1)
    st = torch.cuda.Stream()
    ctx = Context(0, stream=st, precision="fp32_refined")
    ctx.plan_banded([40], rows_per_col=4, window=8, solver=2)
    J = torch.from_numpy(g.standard_normal(40 * 4 * 8).astype(np.float32)).cuda()
    b = torch.from_numpy(g.standard_normal(160).astype(np.float32)).cuda()
    p = torch.empty(40, device="cuda")
    check(torch, late, ctx, st, J, lambda x: ctx.factor_solve(x, b, p, lam=1e-2, refine_steps=1), p)
    ctx.close()


@pytest.mark.parametrize("s", [5, 64])   # a block per thread, and per warp, in the back-substitution
def test_dense(late_input, s):
    torch, late = late_input
    from paper_1802_03773_gb300 import Context, qrkit
    g = np.random.default_rng(2)
    st, K = torch.cuda.Stream(), 60
    ctx = Context(0, stream=st, precision="fp32_refined")
    ctx.plan_blocks(np.full(K, 4), np.full(K, 2), qrkit.COUPLED_DENSE, shared_cols=s)
    t = lambda *n: torch.from_numpy(g.standard_normal(n).astype(np.float32)).cuda()
    J, S, b, N = t(K * 8), t(s, K * 4), t(K * 4), 2 * K + s
    p, q, R = torch.empty(N, device="cuda"), torch.empty(N, device="cuda"), torch.empty(s, s, device="cuda")
    D = t(N).abs() + 0.5
    check(torch, late, ctx, st, D, lambda x: (ctx.factor(J, S, x, 1e-2), ctx.solve(b, p, refine_steps=1)), p)
    check(torch, late, ctx, st, b, lambda x: ctx.solve(x, p, refine_steps=1), p)
    check(torch, late, ctx, st, b, lambda x: ctx.apply_qt(x, q), q)
    check(torch, late, ctx, st, q.clone(), lambda x: ctx.solve_r(x, p), p)
    check(torch, late, ctx, st, q.clone(), lambda x: ctx.solve_blocks(x, p), p[:2 * K])
    sq = t(N).abs().double()
    check(torch, late, ctx, st, sq, lambda x: ctx.norms_from_sumsq(x, p), p)
    ctx.close()


def test_more_and_windows(late_input):
    torch, late = late_input
    from paper_1802_03773_gb300 import Context, qrkit
    g = np.random.default_rng(3)
    st, K, s = torch.cuda.Stream(), 90, 30
    t = lambda *n: torch.from_numpy(g.standard_normal(n).astype(np.float32)).cuda()
    ctx = Context(0, stream=st, precision="fp32")
    ctx.plan_blocks(np.full(K, 6), np.full(K, 3))
    p, qtb = torch.empty(3 * K, device="cuda"), torch.empty(6 * K, device="cuda")
    J, b = t(18 * K), t(6 * K)
    torch.cuda.synchronize()
    ctx.factor_solve(J, b, p, qtb, refine_steps=0)
    ctx.sync_status()
    check(torch, late, ctx, st, qtb, lambda x: ctx.more_solve(x, p, lam=1e-2), p)
    ctx.close()
    ctx = Context(0, stream=st, precision="fp32_refined")
    start = torch.from_numpy(g.integers(0, s - 8, size=K).astype(np.int32)).cuda()
    ctx.plan_blocks(np.full(K, 2), np.full(K, 1), qrkit.COUPLED_WINDOW, shared_cols=s, window=8,
                    window_start=np.zeros(K, dtype=np.int32))
    J, S, b, p = t(2 * K), t(16 * K), t(2 * K), torch.empty(K + s, device="cuda")
    order = torch.zeros(2 * K, device="cuda", dtype=torch.int64)
    check(torch, late, ctx, st, start,
          lambda x: (ctx.set_window_start(x), ctx.factor(J, S, None, 1e-2), ctx.get_row_order(order)), order)
    check(torch, late, ctx, st, b, lambda x: ctx.solve(x, p, refine_steps=1), p)
    ctx.close()


def test_lm(late_input):
    torch, late = late_input
    from paper_1802_03773_gb300 import Context
    g = np.random.default_rng(4)
    st = torch.cuda.Stream()
    ctx = Context(0, stream=st, precision="fp32")
    data = torch.from_numpy(g.standard_normal((50, 2))).cuda()
    ctx.lm_plan([50], [9], data)
    x = torch.from_numpy(np.concatenate([g.random(50) * 6, g.standard_normal(18)])).cuda()
    f, b = torch.empty(100, device="cuda", dtype=torch.float64), torch.empty(100, device="cuda")
    check(torch, late, ctx, st, x, lambda y: ctx.lm_residual(y, f), f)
    check(torch, late, ctx, st, x, lambda y: ctx.lm_linearize(y, b=b), b)
    ctx.close()
