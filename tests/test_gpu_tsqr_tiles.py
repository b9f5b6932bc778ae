"""GPU parity of the register TSQR tiles (dense S without column panels, s <= 64) at the edges of their
variants: 1, 8 / 9, 16 / 17, 32 / 33 and 64 columns (1, 2, 4 or 8 columns per warp), levels of 64, 128 and 256
rows and one more, a last tile with fewer rows than columns, in both precisions, with and without
damping rows, against the FP64 oracle (Secs. 2, 4.2)."""
import numpy as np
import pytest

from oracle import structured as st
from tests.gpu_common import assert_close, cuda_or_skip

pytestmark = pytest.mark.gpu


# columns graded over one decade: the condition number stays below 5e2, so FP64 rounding of a few hundred
# operations per entry (1e-16 each) stays below 1e-11 and float (6e-8 each) below 1e-3
@pytest.mark.parametrize("s,M,lam", [
    (1, 2, 1e-2),       # one reflector of two rows
    (8, 64, 1e-2),      # one tile of the shortest kind, filled
    (9, 65, 0.0),       # the next kind
    (16, 128, 1e-2),
    (17, 129, 0.0),     # a second tile of one row
    (32, 256, 1e-2),    # two tiles of 128 rows: their R rows fill a tile of 64
    (33, 257, 0.0),     # tiles of 256 rows
    (64, 320, 1e-2),
    (24, 1000, 0.0),    # three levels
    (5, 20005, 1e-2),   # more rows than one wave of short tiles takes: 256-row tiles
])
def test_tile_edges(s, M, lam):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, qrkit
    rows = M - s if lam > 0 else M             # rows the blocks leave to the reduced block
    g = np.random.default_rng(11 * s + M)
    each = 5
    K = -(-rows // each)
    left = np.full(K, each)
    left[-1] = rows - each * (K - 1)
    n = left if lam > 0 else left + 1          # blocks n x 1: n rows stay with damping, n - 1 without
    scale = 10.0 ** (np.arange(K + s) / (K + s - 1))
    blocks = [(g.standard_normal((a, 1)) * scale[i]).astype(np.float32) for i, a in enumerate(n)]
    S = (g.standard_normal((int(n.sum()), s)) * scale[K:]).astype(np.float32)
    b = g.standard_normal(int(n.sum())).astype(np.float32)
    off = np.concatenate([[0], np.cumsum(n)])
    P = st.BlockProblem(blocks=[x.astype(np.float64) for x in blocks],
                        coupled=[S[off[i]:off[i + 1]].astype(np.float64) for i in range(K)], s=s,
                        b=b.astype(np.float64), lam=lam)
    p_ref, _ = st.factor_and_solve(P)
    for precision, dt, tol in (("fp64", np.float64, 1e-11), ("fp32", np.float32, 1e-3)):
        J = torch.from_numpy(np.concatenate([x.T.reshape(-1) for x in blocks]).astype(dt)).cuda()
        St = torch.from_numpy(np.ascontiguousarray(S.T).astype(dt)).cuda()
        tb = torch.from_numpy(b.astype(dt)).cuda()
        p = torch.empty(K + s, device="cuda", dtype=tb.dtype)
        ctx = Context(0, precision=precision)
        ctx.plan_blocks(n, np.ones(K), qrkit.COUPLED_DENSE, shared_cols=s)
        ctx.factor(J, St, None, lam)
        ctx.solve(tb, p, refine_steps=0)
        ctx.sync_status()
        assert_close(p.cpu().numpy().astype(np.float64), p_ref, tol)
        ctx.close()
