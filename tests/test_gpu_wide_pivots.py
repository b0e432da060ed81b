"""Inversion in blocks of 512 pivots: sizes around the block and the row count from which it is taken, against fp64 algebra."""
import pytest

from tests.test_gpu_state_products import test_state_matches_fp64_algebra as check_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d1,m,g,k,spread", [
    (3200, 40, 1, 3072, 0.5),      # whole blocks
    (3330, 33, 1, 3073, 1.0),      # one row in the last block
    (3400, 60, 1, 3303, 0.5),      # a last block of 231 rows
    (3600, 50, 9, 345, 0.5),       # groups: one correction step
])
def test_state_with_wide_pivot_blocks(d1, m, g, k, spread):
    check_state(d1, m, g, k, spread)
