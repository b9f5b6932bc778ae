"""Refinement of float plans with windows whose blocks have one shape: residuals 1e9 times what the unknowns explain, and
products that leave the float range (as in test_gpu_large_residuals, whose bounds hold; Secs. 4.2, 5.1)."""
import pytest

from tests.test_gpu_large_residuals import check_large_residual, check_out_of_range

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,K,s,w", [(8, 3, 300, 20, 8), (10, 4, 250, 32, 5)])
def test_large_residual_windows(n, m, K, s, w):
    check_large_residual(n, m, K, s, w)


@pytest.mark.parametrize("n,m,K,s,w", [(8, 3, 60, 20, 8), (10, 4, 50, 32, 5)])
def test_products_out_of_range_windows(n, m, K, s, w):
    check_out_of_range(n, m, K, s, w)
