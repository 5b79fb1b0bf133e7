"""The one-row-per-warp kernel of the approximate path on both sides of the
table size at which its loops are unrolled for fewer columns (320), with the
checks and bars of test_gpu_row_kernel."""
import pytest
from test_gpu_row_kernel import test_row_kernel_matches_oracle as _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_age,n_met", [(20, 4), (50, 6), (32, 10), (107, 3), (27, 12)])
@pytest.mark.parametrize("n", [9, 913])
def test_table_sizes(n_age, n_met, n):
    _check(n_age, n_met, 3, n)
