"""GPU parity, in FP64, of Q_i^T applied to a dense S of fewer columns than a group, and of one more: every shape class
of the kernel, against the oracle (Secs. 4.1, 4.2)."""
import pytest

from tests.test_gpu_dense_block import test_dense_block_apply_matches_oracle as matches_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_hi,m_hi", [(2, 1), (4, 2), (12, 3), (8, 8)])
@pytest.mark.parametrize("s", [1, 2, 3, 5, 9])
def test_partial_groups(n_hi, m_hi, s):
    matches_oracle(130, n_hi, m_hi, s, 1e-3)
