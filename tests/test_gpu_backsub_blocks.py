"""Block back-substitution below and above the block counts from which a thread takes a block instead of a warp: the
block unknowns solve their own least-squares problem for the shared unknowns they were given (Sec. 4.2)."""
import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_refined"])
@pytest.mark.parametrize("s", [15, 16, 21, 30, 63, 64])
@pytest.mark.parametrize("per_sm", [1, 150])   # blocks per SM: by warps (from 16 columns on); by threads (up to 63, doubles 64)
def test_block_unknowns(s, precision, per_sm):
    torch = cuda_or_skip()
    from paper_1802_03773_gb300 import Context, qrkit
    K = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + 3
    g = np.random.default_rng(s + K)
    shape = np.sort(g.integers(0, 3, size=K))[g.permutation(K)]
    n, m = np.array([3, 5, 9])[shape], np.array([1, 3, 5])[shape]
    ro, co = np.concatenate([[0], np.cumsum(n)]), np.concatenate([[0], np.cumsum(m)])
    J = [None] * K
    for i in range(K):
        J[i] = (np.eye(n[i], m[i]) + 0.2 * g.standard_normal((n[i], m[i]))).astype(np.float32)
    S = g.standard_normal((s, int(ro[-1]))).astype(np.float32)   # row c: column c
    b = g.standard_normal(int(ro[-1])).astype(np.float32)
    ctx = Context(0, precision=precision)
    ctx.plan_blocks(n, m, qrkit.COUPLED_DENSE, shared_cols=s)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", ctx.dtype)
    p = torch.empty(int(co[-1]) + s, device="cuda", dtype=ctx.dtype)
    ctx.factor(t(np.concatenate([x.T.reshape(-1) for x in J])), t(S), None, 0.0)
    ctx.solve(t(b), p, refine_steps=1 if precision == "fp32_refined" else 0)
    ctx.sync_status()
    p = p.cpu().numpy().astype(np.float64)
    ctx.close()
    pS = p[co[-1]:]
    rest = b.astype(np.float64) - S.T.astype(np.float64) @ pS
    u = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    for k in range(3):
        idx = np.nonzero(shape == k)[0]
        A = np.stack([J[i] for i in idx]).astype(np.float64)
        rows, cols = ro[idx][:, None] + np.arange(A.shape[1]), co[idx][:, None] + np.arange(A.shape[2])
        x = np.einsum("kij,kj->ki", np.linalg.pinv(A), rest[rows])
        # rounding of the reflectors (8 n m u), of a sum of s products and of b - S p_S before it: a perturbation of the
        # block and of its right-hand side, of which the latter is as large as |b| + |S| |p_S|; first-order bound
        sv = np.linalg.svd(A, compute_uv=False)
        kappa = sv[:, 0] / sv[:, -1]
        size = np.linalg.norm(np.abs(b[rows]) + (np.abs(S.T) @ np.abs(pS))[rows], axis=1)
        bound = u * (8 * A.shape[1] * A.shape[2] + s) * (1 + kappa) ** 2 * size / sv[:, 0]
        assert (np.linalg.norm(p[cols] - x, axis=1) <= bound).all()
