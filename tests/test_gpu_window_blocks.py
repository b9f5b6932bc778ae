"""GPU parity of the per-block kernels for sorted plans of 2 x 1 blocks with windows of 8 (no offset tables, 16-byte
loads of S): block counts around a CTA of 256, with and without damping rows, S on and off the 16-byte
grid (off it the factorization is the general kernel's), against the FP64 oracle (Sec. 4.2)."""
import numpy as np
import pytest

from oracle import structured as st
from tests.gpu_common import assert_close, cuda_or_skip

pytestmark = pytest.mark.gpu


# 200 to 500 rows with N(0, 1) entries: condition number below 1e3 with these sizes, so FP64 stays below 1e-9 and the
# refined float solution below 1e-5
@pytest.mark.parametrize("blocks,cols,lam,shift", [
    ([255], [40], 1e-2, 0),
    ([256], [40], 0.0, 0),
    ([257, 60], [30, 9], 0.0, 0),
    ([257, 60], [30, 9], 1e-2, 1),
    ([257, 60], [30, 9], 0.0, 1),
])
def test_window21_matches_oracle(blocks, cols, lam, shift):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, qrkit
    g = np.random.default_rng(sum(blocks) + shift)
    n, m, w = 2, 1, 8
    K, s = sum(blocks), sum(cols)
    c0 = np.concatenate([[0], np.cumsum(cols)])
    start = np.concatenate([c0[k] + g.integers(0, cols[k], size=b) for k, b in enumerate(blocks)])
    end = np.concatenate([np.full(b, c0[k + 1]) for k, b in enumerate(blocks)])
    J = g.standard_normal((K, n, m))
    S = g.standard_normal((K, n, w))
    S[np.broadcast_to((start[:, None] + np.arange(w) >= end[:, None])[:, None, :], S.shape)] = 0.0
    b = g.standard_normal(K * n)
    J, S, b = (x.astype(np.float32).astype(np.float64) for x in (J, S, b))
    dense = [np.zeros((n, s)) for _ in range(K)]
    for i in range(K):
        k = min(w, s - start[i])
        dense[i][:, start[i]:start[i] + k] = S[i][:, :k]
    P = st.BlockProblem(blocks=list(J), coupled=dense, s=s, b=b, lam=lam)
    p_ref, _ = st.factor_and_solve(P)
    for precision, steps, tol in (("fp64", 0, 1e-9), ("fp64", 1, 1e-9), ("fp32_refined", 2, 1e-5)):
        ctx = Context(0, precision=precision)
        dt = ctx.dtype
        ctx.plan_blocks(np.full(K, n), np.full(K, m), qrkit.COUPLED_WINDOW, shared_cols=s, window=w, window_start=start,
                        segment_cols=cols, segment_blocks=blocks)
        tJ = torch.from_numpy(np.ascontiguousarray(J.transpose(0, 2, 1)).reshape(-1)).to("cuda", dt)
        tS = torch.empty(S.size + shift, device="cuda", dtype=dt)[shift:]
        tS.copy_(torch.from_numpy(np.ascontiguousarray(S.transpose(0, 2, 1)).reshape(-1)))
        ctx.factor(tJ, tS, None, lam)
        p = torch.empty(K * m + s, device="cuda", dtype=dt)
        ctx.solve(torch.from_numpy(b).to("cuda", dt), p, refine_steps=steps)
        ctx.sync_status()
        assert_close(p.cpu().numpy().astype(np.float64), p_ref, tol)
        ctx.close()
