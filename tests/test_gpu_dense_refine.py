"""GPU parity of the refinement step and the solves of float plans with a dense S: uneven blocks, row
counts off and on the 16-byte grid, chunk edges of the row, block and column passes, and an S whose
address is not 16-byte aligned, against the FP64 oracle (Secs. 4.1, 4.2, 5.1)."""
import numpy as np
import pytest

from oracle import structured as st
from tests.gpu_common import assert_close, cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,s,rows,shift", [
    (9, 3, None, 0),          # fewer columns than a CTA's warps
    (40, 15, None, 0),        # the last s solved by a thread per block
    (40, 16, None, 1),        # the first s solved by a warp per block; S off the 16-byte grid
    (41, 17, None, 0),        # s not a multiple of 4
    (370, 33, 2048, 0),       # rows fill one chunk of the column sums exactly
    (371, 64, 2052, 3),       # a second chunk of 4 rows; S off the 16-byte grid
    (300, 96, 1501, 0),       # an odd row count: 4-byte loads
])
def test_refined_dense_solve_matches_oracle(K, s, rows, shift):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, qrkit
    g = np.random.default_rng(100 * K + s)
    m = g.integers(1, 5, size=K)
    n = m + g.integers(1, 6, size=K)
    if rows is not None:   # move rows one at a time until the total is the one asked for
        i = 0
        while n.sum() != rows:
            step = 1 if n.sum() < rows else -1
            if m[i % K] < n[i % K] + step <= 12:
                n[i % K] += step
            i += 1
    scale = 10.0 ** (np.arange(int(m.sum()) + s) / (m.sum() + s - 1))
    blocks, c0 = [], 0
    for a, c in zip(n, m):
        blocks.append((g.standard_normal((a, c)) * scale[c0:c0 + c]).astype(np.float32))
        c0 += c
    S = (g.standard_normal((int(n.sum()), s)) * scale[c0:]).astype(np.float32)
    b = g.standard_normal(int(n.sum())).astype(np.float32)
    off = np.concatenate([[0], np.cumsum(n)])
    P = st.BlockProblem(blocks=[x.astype(np.float64) for x in blocks],
                        coupled=[S[off[i]:off[i + 1]].astype(np.float64) for i in range(K)], s=s,
                        b=b.astype(np.float64), lam=1e-2)
    p_ref, _ = st.factor_and_solve(P)
    ctx = Context(0, precision="fp32_refined")
    ctx.plan_blocks(n, m, qrkit.COUPLED_DENSE, shared_cols=s)
    J = torch.from_numpy(np.concatenate([x.T.reshape(-1) for x in blocks])).cuda()
    St = torch.empty(S.size + shift, device="cuda", dtype=torch.float32)[shift:]
    St.copy_(torch.from_numpy(np.ascontiguousarray(S.T).reshape(-1)))
    ctx.factor(J, St, None, 1e-2)
    p = torch.empty(c0 + s, device="cuda", dtype=torch.float32)
    ctx.solve(torch.from_numpy(b).cuda(), p, refine_steps=2)
    ctx.sync_status()
    assert_close(p.cpu().numpy().astype(np.float64), p_ref, 1e-6)
    ctx.close()
