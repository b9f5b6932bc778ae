"""GPU parity, in FP64, of Q_i^T applied to a dense S through shared-memory column segments: block
counts around the 128 of a CTA, every shape class of the kernel, odd row counts, column counts that
leave a partial group, with and without damping rows, against the oracle (Secs. 4.1, 4.2)."""
import numpy as np
import pytest

from oracle import structured as st
from tests.gpu_common import assert_close, cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,n_hi,m_hi,s,lam", [
    (127, 2, 1, 5, 1e-3),      # at most 3 x 1 augmented
    (128, 4, 2, 8, 1e-3),      # at most 6 x 2 augmented, one full CTA
    (129, 4, 2, 9, 0.0),       # a second CTA of one block; blocks as wide as tall leave no rows
    (130, 12, 3, 13, 1e-3),
    (131, 13, 3, 4, 0.0),
    (140, 8, 8, 31, 1e-3),     # 16 augmented rows, 8 columns
    (260, 16, 8, 33, 0.0),
])
def test_dense_block_apply_matches_oracle(K, n_hi, m_hi, s, lam):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, qrkit
    g = np.random.default_rng(1000 * K + s)
    m = g.integers(1, m_hi + 1, size=K)
    n = np.array([g.integers(c, n_hi + 1) for c in m])
    n[0] = min(n_hi, 16 - m[0] if lam > 0 else 16)
    if lam > 0:
        n = np.minimum(n, 16 - m)
    blocks = [g.standard_normal((a, c)) for a, c in zip(n, m)]
    S, b = g.standard_normal((int(n.sum()), s)), g.standard_normal(int(n.sum()))
    off = np.concatenate([[0], np.cumsum(n)])
    P = st.BlockProblem(blocks=blocks, coupled=[S[off[i]:off[i + 1]] for i in range(K)], s=s, b=b, lam=lam)
    p_ref, _ = st.factor_and_solve(P)
    ctx = Context(0, precision="fp64")
    ctx.plan_blocks(n, m, qrkit.COUPLED_DENSE, shared_cols=s)
    ctx.factor(torch.from_numpy(np.concatenate([x.T.reshape(-1) for x in blocks])).cuda(),
               torch.from_numpy(np.ascontiguousarray(S.T)).cuda(), None, lam)
    p = torch.empty(int(m.sum()) + s, device="cuda", dtype=torch.float64)
    ctx.solve(torch.from_numpy(b).cuda(), p, refine_steps=0)
    ctx.sync_status()
    # square random blocks reach condition numbers of a few thousand: 1e-9 leaves them room in FP64
    assert_close(p.cpu().numpy(), p_ref, 1e-9)
    ctx.close()
