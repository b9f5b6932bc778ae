"""Re-tuning a banded plan while solves are queued on a stream that does not wait for the default one, and
replaying a captured solve after re-tuning: bit for bit what a context of its own gives for each strategy (the
compression's tables of a strategy are never overwritten)."""
import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu

CHOICES = ["compress 0 2", "compress 0 64", "compress 1 1", "compress 0 5", "compress 0 17"]


def test_retuning_beside_queued_and_captured_solves():
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context
    g = np.random.default_rng(5)
    cols, rpc = [3000, 50, 701, 8], 40
    N = sum(cols)
    J = torch.from_numpy(g.standard_normal((N * rpc, 8)).astype(np.float32).reshape(-1)).cuda()
    b = torch.from_numpy(g.standard_normal(N * rpc).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    solve = lambda ctx, p: ctx.factor_solve(J, b, p, lam=1e-2, refine_steps=1)

    want = []
    for choice in CHOICES:
        ctx = Context(0, precision="fp32_refined")
        ctx.plan_banded(cols, rows_per_col=rpc, window=8, solver=2)
        ctx.apply_tuning(choice)
        p = torch.empty(N, device="cuda")
        solve(ctx, p)
        ctx.sync_status()
        want.append(p)
        ctx.close()

    stream = torch.cuda.Stream()
    ctx = Context(0, stream=stream, precision="fp32_refined")
    ctx.plan_banded(cols, rows_per_col=rpc, window=8, solver=2)
    out = [torch.empty(N, device="cuda") for _ in range(4 * len(CHOICES))]
    held = torch.empty(N, device="cuda")
    torch.cuda.synchronize()
    for k, p in enumerate(out):   # no synchronization between a solve and the next strategy
        ctx.apply_tuning(CHOICES[k % len(CHOICES)])
        solve(ctx, p)
    ctx.sync_status()
    for k, p in enumerate(out):
        assert torch.equal(p, want[k % len(CHOICES)]), CHOICES[k % len(CHOICES)]

    ctx.apply_tuning(CHOICES[0])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        solve(ctx, held)
    for choice, ref in zip(CHOICES, want):
        ctx.apply_tuning(choice)
        solve(ctx, out[0])
        with torch.cuda.stream(stream):
            graph.replay()
        ctx.sync_status()
        assert torch.equal(out[0], ref) and torch.equal(held, want[0])
        held.zero_()
        torch.cuda.synchronize()
    graph.reset()
    ctx.close()
