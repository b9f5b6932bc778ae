"""GPU parity of windowed plans whose blocks all have one shape (sorted as blocks before the factorization,
column sums by sorted runs): shape classes of the kernels, block counts around a sort chunk of 256 and a run
of 32, segments without a full window, windows narrower than 8, with and without damping, against the FP64
oracle; the row order against a stable sort (Secs. 4.2, 4.3)."""
import numpy as np
import pytest

from oracle import structured as st
from tests.gpu_common import assert_close, cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,w,blocks,cols,lam", [
    (2, 1, 8, [257], [40], 1e-2),               # one block past a chunk
    (2, 1, 8, [256, 31, 33], [30, 8, 9], 1e-2), # several segments, runs that end inside one
    (2, 1, 5, [100, 7], [12, 5], 1e-2),
    (4, 2, 8, [70, 65], [20, 11], 0.0),         # without damping rows: n - m reduced rows per block
    (7, 3, 6, [64, 50], [17, 9], 1e-2),         # the general class
])
def test_uniform_windows_match_oracle(n, m, w, blocks, cols, lam):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, qrkit
    g = np.random.default_rng(10 * n + w)
    K, s = sum(blocks), sum(cols)
    c0 = np.concatenate([[0], np.cumsum(cols)])
    start = np.concatenate([c0[k] + g.integers(0, cols[k], size=b) for k, b in enumerate(blocks)])
    end = np.concatenate([np.full(b, c0[k + 1]) for k, b in enumerate(blocks)])
    J = g.standard_normal((K, n, m))
    S = g.standard_normal((K, n, w))
    S[np.broadcast_to((start[:, None] + np.arange(w) >= end[:, None])[:, None, :], S.shape)] = 0.0
    b = g.standard_normal(K * n)
    J, S, b = (x.astype(np.float32).astype(np.float64) for x in (J, S, b))
    # a window may reach past the last column (with zeros): the oracle is given dense rows
    dense = [np.zeros((n, s)) for _ in range(K)]
    for i in range(K):
        k = min(w, s - start[i])
        dense[i][:, start[i]:start[i] + k] = S[i][:, :k]
    P = st.BlockProblem(blocks=list(J), coupled=dense, s=s, b=b, lam=lam)
    p_ref, _ = st.factor_and_solve(P)
    rows = n if lam > 0 else n - m
    for precision, steps, tol in (("fp64", 0, 1e-9), ("fp64", 1, 1e-9), ("fp32_refined", 2, 1e-5)):
        ctx = Context(0, precision=precision)
        dt = ctx.dtype
        ctx.plan_blocks(np.full(K, n), np.full(K, m), qrkit.COUPLED_WINDOW, shared_cols=s, window=w, window_start=start,
                        segment_cols=cols, segment_blocks=blocks)
        tJ = torch.from_numpy(np.ascontiguousarray(J.transpose(0, 2, 1)).reshape(-1)).to("cuda", dt)
        tS = torch.from_numpy(np.ascontiguousarray(S.transpose(0, 2, 1)).reshape(-1)).to("cuda", dt)
        ctx.factor(tJ, tS, None, lam)
        p = torch.empty(K * m + s, device="cuda", dtype=dt)
        ctx.solve(torch.from_numpy(b).to("cuda", dt), p, refine_steps=steps)
        order = torch.empty(K * rows, device="cuda", dtype=torch.int64)
        ctx.get_row_order(order)
        ctx.sync_status()
        assert_close(p.cpu().numpy().astype(np.float64), p_ref, tol)
        key = np.repeat(start, rows)   # segments own ascending column ranges, so the start is the whole key
        np.testing.assert_array_equal(order.cpu().numpy(), np.argsort(key, kind="stable"))
        ctx.close()
