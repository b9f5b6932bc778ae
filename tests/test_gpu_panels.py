"""GPU parity of the column-panel TSQR (float dense S, s a multiple of 32, tiles of 1024 rows) at the
edges of its tiles: levels of 256, 512 and 1024 rows and four more, a last tile of four rows, row
counts that need padding, with and without damping rows, against the FP64 oracle (Secs. 2, 4.2)."""
import numpy as np
import pytest

from oracle import structured as st
from tests.gpu_common import assert_close, cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,M,lam", [
    (64, 256, 1e-2),     # one tile of the shortest kind, filled
    (64, 260, 1e-2),     # the next kind
    (96, 512, 0.0),
    (96, 515, 0.0),      # padded by one zero row
    (64, 1024, 1e-2),    # one full tile
    (64, 1028, 1e-2),    # a second tile of four rows: fewer rows than the panel has columns
    (128, 1055, 0.0),    # 31 rows in the second tile, padded to 32
    (160, 3071, 1e-2),   # three tiles; the later panels' levels end 32 rows shorter each
])
def test_panel_tile_edges(s, M, lam):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, qrkit
    rows = M - s if lam > 0 else M             # rows the blocks leave to the reduced block
    g = np.random.default_rng(7 * s + M)
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
    J = torch.from_numpy(np.concatenate([x.T.reshape(-1) for x in blocks])).cuda()
    St = torch.from_numpy(np.ascontiguousarray(S.T)).cuda()
    tb = torch.from_numpy(b).cuda()
    p = torch.empty(K + s, device="cuda", dtype=torch.float32)
    for precision, steps, tol in (("fp32", 0, 1e-4), ("fp32_refined", 2, 1e-6)):
        ctx = Context(0, precision=precision)
        ctx.plan_blocks(n, np.ones(K), qrkit.COUPLED_DENSE, shared_cols=s)
        ctx.factor(J, St, None, lam)
        ctx.solve(tb, p, refine_steps=steps)
        ctx.sync_status()
        assert_close(p.cpu().numpy().astype(np.float64), p_ref, tol)
        ctx.close()
