"""Squared residuals of banded float plans for right-hand sides of any scale: the solution is linear in b, which the
factorization never squares, and res2 is a double (Sec. 4.4)."""
import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip
from tests.test_gpu_banded import batch, oracle_solutions

pytestmark = pytest.mark.gpu


# the bound of an unscaled system: float rounding errors of some ten operations (6e-7) in every entry of the residual
@pytest.mark.parametrize("tuning", [None, "compress 0 4"])
@pytest.mark.parametrize("scale", [1e-30, 1e-25, 1e-16, 1e-14, 1.0, 1e14, 1e20, 1e30])
def test_squared_residual_of_scaled_rhs(scale, tuning):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context
    cols, rpc = [200, 9, 40], 5
    inst, vals, b = batch(cols, rpc, 8, np.float32, seed=3)
    b = (b * np.float32(scale)).astype(np.float32)
    off = np.concatenate([[0], np.cumsum([rpc * n for n in cols])])
    inst = [dict(d, b=b[off[k]:off[k + 1]].astype(np.float64) / scale) for k, d in enumerate(inst)]
    x, _, want = oracle_solutions(inst, 1e-2)
    ctx = Context(0, precision="fp32")
    ctx.plan_banded(cols, rows_per_col=rpc, window=8, solver=2)
    if tuning:
        ctx.apply_tuning(tuning)
    p = torch.empty(sum(cols), device="cuda")
    ctx.factor_solve(torch.from_numpy(np.ascontiguousarray(vals.reshape(-1))).cuda(), torch.from_numpy(b).cuda(), p,
                     lam=1e-2, refine_steps=0)
    ctx.sync_status()
    res2 = np.zeros(len(cols))
    ctx.get_band_factor(None, None, res2)
    ctx.close()
    got = p.cpu().numpy().astype(np.float64) / scale
    assert np.linalg.norm(got - x) <= 1e-5 * np.linalg.norm(x)
    np.testing.assert_allclose(res2 / scale / scale, want, rtol=2e-6)


# A power of two scales every operation exactly, so the solution of a scaled J is the inversely scaled one, but for
# the entries that underflow against the others: rounding errors of plain float
@pytest.mark.parametrize("rpc,tuning", [(4, None), (4, "compress 0 3"), (25, None)])
@pytest.mark.parametrize("power", [-62, -60, -57, -52, 50, 56])
def test_scaled_matrix(power, rpc, tuning):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context
    N = 200
    inst, vals, b = batch([N], rpc, 8, np.float32, seed=7)
    J, rhs = torch.from_numpy(np.ascontiguousarray(vals.reshape(-1))).cuda(), torch.from_numpy(b).cuda()

    def solve(factor):
        ctx = Context(0, precision="fp32")
        ctx.plan_banded([N], rows_per_col=rpc, window=8, solver=2)
        if tuning:
            ctx.apply_tuning(tuning)
        p = torch.empty(N, device="cuda")
        ctx.factor_solve(J * factor, rhs, p, lam=0.5, refine_steps=0)
        ctx.sync_status()
        ctx.close()
        return p.cpu().numpy().astype(np.float64) * factor

    want = solve(1.0)
    assert np.abs(solve(2.0 ** power) - want).max() <= 1e-6 * np.abs(want).max()
