"""Block back-substitution in place: qrkit_solve_r and qrkit_solve_blocks with p the same buffer as qtb give what
separate buffers give (Sec. 5.1)."""
import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("s", [5, 16, 30, 64])   # a block per thread, and per warp
def test_in_place(s, precision):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, qrkit
    g = np.random.default_rng(s)
    K = 5000
    m = g.integers(1, 8, size=K)
    n = m + g.integers(0, 9 - m)
    ctx = Context(0, precision=precision)
    ctx.plan_blocks(n, m, qrkit.COUPLED_DENSE, shared_cols=s)
    t = lambda *size: torch.from_numpy(g.standard_normal(size)).to("cuda", ctx.dtype)
    N = int(m.sum()) + s
    ctx.factor(t(int((n * m).sum())), t(s, int(n.sum())), None, 1e-2)
    b, q, p = t(int(n.sum())), torch.empty(N, device="cuda", dtype=ctx.dtype), torch.empty(N, device="cuda", dtype=ctx.dtype)
    ctx.apply_qt(b, q)
    ctx.solve_r(q, p)
    r = q.clone()
    ctx.solve_r(r, r)
    ctx.sync_status()
    assert torch.equal(r, p)
    r = q.clone()
    r[N - s:] = p[N - s:]
    ctx.solve_blocks(r, r)
    ctx.sync_status()
    assert torch.equal(r, p)
    ctx.close()
