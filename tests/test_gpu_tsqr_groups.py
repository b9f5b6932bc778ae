"""GPU parity of the register TSQR tiles at every count of column groups of eight that a warp set takes in
double (1 to 8), the last group one column, all but one and full, against the FP64 oracle (Secs. 2, 4.2)."""
import pytest

from tests.test_gpu_tsqr_tiles import test_tile_edges as tile_edges

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [64, 128, 300])   # tiles of 64, 128 and 256 rows
@pytest.mark.parametrize("s", [c for g in range(8) for c in (8 * g + 1, 8 * g + 7, 8 * g + 8)])
def test_column_groups(s, M):
    if M > s:
        tile_edges(s, M, 1e-2)
