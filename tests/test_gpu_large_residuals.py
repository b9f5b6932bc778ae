"""Refinement of float plans whose residual is 1e9 times what the unknowns explain: the gradient J^T r is then the
cancellation of products a billion times its size, which only sums as accurate as in double resolve; and
right-hand sides whose products with J leave the float range (Secs. 4.2, 5.1)."""
import numpy as np
import pytest

from tests.gpu_common import cuda_or_skip

pytestmark = pytest.mark.gpu


def system(n, m, K, s, w, seed):
    """Blocks n x m, a dense S (w = 0) or windows of w, values rounded to float; the whole matrix and its pieces."""
    g = np.random.default_rng(seed)
    f = lambda *size: g.standard_normal(size).astype(np.float32).astype(np.float64)
    J, A = f(K, n, m), np.zeros((K * n, K * m + s))
    start = None
    if w == 0:
        S = f(K * n, s)
        A[:, K * m:] = S
    else:
        S, start = f(K, n, w), g.integers(0, s - w + 1, size=K)
    for i in range(K):
        A[i * n:(i + 1) * n, i * m:(i + 1) * m] = J[i]
        if w:
            A[i * n:(i + 1) * n, K * m + start[i]:K * m + start[i] + w] = S[i]
    return A, J, S, start, g


def refined(torch, n, m, K, s, w, J, S, start, b, lam, steps):
    from paper_1802_03773_gb300 import Context, qrkit
    ctx = Context(0, precision="fp32_refined")
    if w:
        ctx.plan_blocks(np.full(K, n), np.full(K, m), qrkit.COUPLED_WINDOW, shared_cols=s, window=w, window_start=start)
        tS = np.ascontiguousarray(S.transpose(0, 2, 1)).reshape(-1)
    else:
        ctx.plan_blocks(np.full(K, n), np.full(K, m), qrkit.COUPLED_DENSE, shared_cols=s)
        tS = np.ascontiguousarray(S.T)
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x).astype(np.float32)).cuda()
    p = torch.empty(K * m + s, device="cuda")
    ctx.factor(t(J.transpose(0, 2, 1).reshape(-1)), t(tS), None, lam)
    ctx.solve(t(b), p, refine_steps=steps)
    ctx.sync_status()
    ctx.close()
    return p.cpu().numpy().astype(np.float64)


def solution(A, b, lam):
    D = np.linalg.norm(A, axis=0)
    D[D == 0] = 1.0   # an untouched shared column
    return np.linalg.solve(A.T @ A + lam * np.diag(D * D), A.T @ b)


# The entries of p are floats: 2^-24 = 6e-8.  The gradient in double, with 1e3 products of a residual of 1e9 per column, is
# off by 1e9 sqrt(1e3) 2^-53 = 4e-6 in sums whose system has 1e3 on its diagonal: 4e-9 in p.  Together below 7e-8
@pytest.mark.parametrize("n,m,K,s,w", [(8, 3, 300, 20, 0), (10, 4, 250, 32, 0)])
def test_large_residual_dense(n, m, K, s, w):
    check_large_residual(n, m, K, s, w)


def check_large_residual(n, m, K, s, w):
    torch = cuda_or_skip()
    A, J, S, start, g = system(n, m, K, s, w, seed=n)
    Q = np.linalg.qr(A)[0]
    r = g.standard_normal(A.shape[0])
    for _ in range(3):
        r -= Q @ (Q.T @ r)
    b = (A @ (30.0 * g.standard_normal(A.shape[1])) + 1e9 * r).astype(np.float32).astype(np.float64)
    # the normal equations in long double arithmetic: A^T b cancels, too
    D = np.linalg.norm(A, axis=0)
    rhs = (A.T.astype(np.longdouble) @ b.astype(np.longdouble)).astype(np.float64)
    x = np.linalg.solve(A.T @ A + 1e-3 * np.diag(D * D), rhs)
    p = refined(torch, n, m, K, s, w, J, S, start, b, 1e-3, 6)
    assert np.linalg.norm(p - x) <= 7e-8 * np.linalg.norm(x)
    assert np.linalg.norm(p[K * m:] - x[K * m:]) <= 7e-8 * np.linalg.norm(x[K * m:])


# A scaled b scales the solution, whatever the products in between: 2^-22 of its largest entry
@pytest.mark.parametrize("n,m,K,s,w", [(8, 3, 60, 20, 0), (10, 4, 50, 32, 0)])
def test_products_out_of_range_dense(n, m, K, s, w):
    check_out_of_range(n, m, K, s, w)


def check_out_of_range(n, m, K, s, w):
    torch = cuda_or_skip()
    A, J, S, start, g = system(n, m, K, s, w, seed=100 + n)
    J, S = J * 2.0 ** 40, S * 2.0 ** 40
    b = g.standard_normal(A.shape[0]).astype(np.float32).astype(np.float64)
    want = solution(A, b, 1e-2)
    p = refined(torch, n, m, K, s, w, J, S, start, b * 2.0 ** 90, 1e-2, 2) / 2.0 ** 50
    assert np.abs(p - want).max() <= 2.0 ** -22 * np.abs(want).max()
