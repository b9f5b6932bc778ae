"""Squared column sums of float plans, which are doubles: as accurate as sums in double at every scale that float
values have, for a dense S, and through the damped solve for a windowed S whose blocks are sorted (Secs. 4.2,
5.2)."""
import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu

SCALES = [1e-36, 1e-30, 1e-23, 1e-21, 1e-15, 1.0, 1e15, 1e19, 1e30]


# one rounding per thread's sum and one per addition in double: 5 lanes, 8 warps and 3 chunks in a column's longest chain
@pytest.mark.parametrize("scale", SCALES)
def test_dense_column_sums(scale):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, qrkit
    g = np.random.default_rng(1)
    K, n, m, s = 5000, 4, 2, 9
    J = g.standard_normal(K * n * m).astype(np.float32)
    S = (g.standard_normal((s, K * n)) * scale).astype(np.float32)
    S[0] = 0.0                          # a zero column
    S[1, ::2] *= np.float32(1e-10)      # two sizes in one column
    S[2, 5:] = 0.0                      # few entries
    ctx = Context(0, precision="fp32")
    ctx.plan_blocks(np.full(K, n), np.full(K, m), qrkit.COUPLED_DENSE, shared_cols=s)
    sq = torch.empty(K * m + s, device="cuda", dtype=torch.float64)
    ctx.column_sumsq(torch.from_numpy(J).cuda(), torch.from_numpy(S).cuda(), sq)
    ctx.sync_status()
    ctx.close()
    got = sq[K * m:].cpu().numpy()
    want = np.array([np.sum(row.astype(np.longdouble) ** 2) for row in S])
    assert got[0] == 0.0
    assert (np.abs(got[1:] - want[1:]) / want[1:]).max() <= 20 * 2.0 ** -53


# Scaling S's columns scales their norms, so the damped solution's shared unknowns scale inversely and the others stay: with
# a power of two, in every bit of what is computed
@pytest.mark.parametrize("power", [-60, -52, 50])
def test_window_norms_scale(power):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, qrkit
    g = np.random.default_rng(2)
    K, s = 300, 24
    start = g.integers(0, s - 8, size=K)
    J = torch.from_numpy(g.standard_normal(2 * K).astype(np.float32)).cuda()
    S = torch.from_numpy(g.standard_normal(16 * K).astype(np.float32)).cuda()
    b = torch.from_numpy(g.standard_normal(2 * K).astype(np.float32)).cuda()

    def solve(factor):
        ctx = Context(0, precision="fp32")
        ctx.plan_blocks(np.full(K, 2), np.full(K, 1), qrkit.COUPLED_WINDOW, shared_cols=s, window=8, window_start=start)
        p = torch.empty(K + s, device="cuda")
        ctx.factor(J, S * factor, None, 0.5)
        ctx.solve(b, p, refine_steps=0)
        ctx.sync_status()
        ctx.close()
        return p.cpu().numpy().astype(np.float64)

    p, q = solve(1.0), solve(2.0 ** power)
    q[K:] *= 2.0 ** power
    np.testing.assert_allclose(q, p, rtol=1e-5, atol=1e-5 * np.abs(p).max())
