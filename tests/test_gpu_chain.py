"""Launches that begin while the kernel before them ends: queued block solves, without a synchronization between
them, give bit for bit what separate contexts give one at a time, eagerly and replayed from a CUDA graph.  Plans
whose narrow and wide tasks run side by side, plans with one class only, and one too large for it."""
import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,cols", [(1, (1, 6)), (40, (1, 4)), (40, (5, 6)), (500, (1, 6)), (3000, (1, 6)),
                                    (40000, (1, 6))])
def test_queued_block_solves_are_the_same(K, cols):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context
    g = np.random.default_rng(17 * K + cols[0])
    m = g.integers(cols[0], cols[1] + 1, size=K)
    n = np.minimum(16, m + g.integers(0, 11, size=K))
    values, rows, unknowns = int((n * m).sum()), int(n.sum()), int(m.sum())
    data = [(torch.from_numpy(g.standard_normal(values).astype(np.float32)).cuda(),
             torch.from_numpy(g.standard_normal(rows).astype(np.float32)).cuda()) for _ in range(4)]

    want = []
    for J, b in data:
        ctx = Context(0, precision="fp32_refined")
        ctx.plan_blocks(n, m)
        p = torch.empty(unknowns, device="cuda")
        torch.cuda.synchronize()
        ctx.factor_solve(J, b, p, refine_steps=2)
        ctx.sync_status()
        want.append(p)
        ctx.close()

    stream = torch.cuda.Stream()
    ctx = Context(0, stream=stream, precision="fp32_refined")
    ctx.plan_blocks(n, m)
    J, b, p = torch.zeros_like(data[0][0]), torch.zeros_like(data[0][1]), torch.empty(unknowns, device="cuda")
    torch.cuda.synchronize()
    solve = lambda: ctx.factor_solve(J, b, p, refine_steps=2)

    def queue(step):
        out = []
        with torch.cuda.stream(stream):
            for Ji, bi in data:
                J.copy_(Ji)
                b.copy_(bi)
                step()
                out.append(p.clone())
        stream.synchronize()
        return out

    for got, ref in zip(queue(solve), want):
        assert torch.equal(got, ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        solve()
    for got, ref in zip(queue(graph.replay), want):
        assert torch.equal(got, ref)
    ctx.sync_status()
    ctx.close()
