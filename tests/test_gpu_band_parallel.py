"""GPU parity of the parallel banded QR at the edges of its work split: block counts around the 128 that
an instance's one-CTA tail takes, several batch levels, rows per column that fill a step of four rows or do
not, narrow windows, row groups too large to stage, a J off the 16-byte grid, and every merge depth of the
split compression, against the FP64 oracle (Sec. 4.4)."""
import numpy as np
import pytest

from tests.gpu_common import assert_close, cuda_or_skip
from tests.test_gpu_banded import batch, oracle_solutions

pytestmark = pytest.mark.gpu


def solve(cols, rpc, w, precision, lam, shift=0, tuning=None, refine_steps=2):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context
    dtype = np.float64 if precision == "fp64" else np.float32
    inst, vals, b = batch(cols, rpc, w, dtype, seed=31)
    ctx = Context(0, precision=precision)
    ctx.plan_banded(cols, rows_per_col=rpc, window=w, solver=2)
    if tuning:
        ctx.apply_tuning(tuning)
    J = torch.empty(vals.size + shift, device="cuda", dtype=ctx.dtype)[shift:]
    J.copy_(torch.from_numpy(np.ascontiguousarray(vals.reshape(-1))))
    p = torch.empty(int(np.sum(cols)), device="cuda", dtype=ctx.dtype)
    ctx.factor_solve(J, torch.from_numpy(b).cuda(), p, None, lam=lam, refine_steps=refine_steps)
    ctx.sync_status()
    res2 = np.zeros(len(cols))
    ctx.get_band_factor(None, None, res2)
    ctx.close()
    return p.cpu().numpy().astype(np.float64), res2, inst


@pytest.mark.parametrize("cols,rpc,w,shift", [
    ([1016, 1017, 1024, 1025, 3], 3, 8, 0),   # 127, 128, 128 and 129 blocks: no level, and one, before the tail
    ([2041, 8, 2056], 2, 8, 1),               # 256 and 257 blocks; J off the 16-byte grid
    ([9, 260, 1], 5, 8, 0),                   # five rows per column: a step of four and one of one
    ([200, 31], 1, 7, 0),                     # one row per column, odd rows
    ([130, 50], 3, 1, 0),                     # a window of one column
    ([70, 9], 90, 8, 0),                      # 720 values per column: groups read from global memory
])
def test_parallel_matches_oracle(cols, rpc, w, shift):
    p, res2, inst = solve(cols, rpc, w, "fp64", 1e-2, shift)
    x, _, r2 = oracle_solutions(inst, 1e-2)
    np.testing.assert_allclose(p, x, rtol=1e-11, atol=1e-11 * np.abs(x).max())
    np.testing.assert_allclose(res2, r2, rtol=1e-9)
    p, _, inst = solve(cols, rpc, w, "fp32_refined", 1e-2, shift)
    x, _, _ = oracle_solutions(inst, 1e-2)
    assert_close(p, x, 1e-6)


@pytest.mark.parametrize("splits", [2, 4, 5, 16, 17, 64])
def test_split_compression_matches_oracle(splits):
    p, res2, inst = solve([40, 17], 11, 8, "fp64", 1e-2, tuning=f"compress 0 {splits}")
    x, _, r2 = oracle_solutions(inst, 1e-2)
    np.testing.assert_allclose(p, x, rtol=1e-11, atol=1e-11 * np.abs(x).max())
    np.testing.assert_allclose(res2, r2, rtol=1e-9)


def test_many_instances_of_mixed_depth():
    """Instances whose compressed block rows share lines with instances that are levels ahead of them."""
    g = np.random.default_rng(4)
    cols = list(g.integers(1, 40, size=300)) + [1100, 2100, 5, 1030] + list(g.integers(200, 900, size=40))
    p, _, inst = solve(cols, 4, 8, "fp32_refined", 1e-3)
    x, _, _ = oracle_solutions(inst, 1e-3)
    assert_close(p, x, 1e-6)
