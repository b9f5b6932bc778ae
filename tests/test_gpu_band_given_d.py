"""Banded float plans with a given D: the refined solution's fixed point is that of the D and lambda of this call, for
D far from the column norms, lambda of any size that D balances, and calls with and without D in turn
(Secs. 4.4, 5.2)."""
import numpy as np
import pytest

from tests.gpu_common import assert_close, cuda_or_skip
from tests.test_gpu_banded import batch, oracle_solutions

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam,size", [(1e-2, 1.0), (1e-2, 1e3), (1e-44, 1e22), (1e-50, 3e24), (1e40, 1e-20), (1e-12, 1e6)])
def test_given_d(lam, size):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context
    cols, rpc = [120, 9], 4
    inst, vals, b = batch(cols, rpc, 8, np.float32, seed=11)
    N = sum(cols)
    g = np.random.default_rng(3)
    D = (size * 10.0 ** g.uniform(-1.5, 1.5, N)).astype(np.float32)   # graded over three decades
    ctx = Context(0, precision="fp32_refined")
    ctx.plan_banded(cols, rows_per_col=rpc, window=8, solver=2)
    J, rhs = torch.from_numpy(np.ascontiguousarray(vals.reshape(-1))).cuda(), torch.from_numpy(b).cuda()
    p = torch.empty(N, device="cuda")
    for use in (None, D, None):
        # the column norms with an ordinary lambda, before and after: neither call's D may reach the other
        lam_now = 1e-2 if use is None else lam
        ctx.factor_solve(J, rhs, p, None, D=None if use is None else torch.from_numpy(use).cuda(), lam=lam_now,
                         refine_steps=4)
        ctx.sync_status()
        want, _, _ = oracle_solutions(inst, lam_now, None if use is None else use.astype(np.float64))
        assert_close(p.cpu().numpy().astype(np.float64), want, 1e-6)
    ctx.close()
