"""List builds on both sides of the sizes where the slices change (8, 16 and 32
atoms a warp at 24,576 and 49,152 atoms), as test_gpu_list_build: every entry
against the oracle, and half lists hold one of each mirror pair."""
import pytest

from test_gpu_list_build import test_lists_equal_the_oracle as lists_equal_the_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L", [(24575, 80.0), (24576, 80.0), (49151, 100.0), (49152, 100.0)])
def test_both_sides(mdk, ora, n, L):
    lists_equal_the_oracle(mdk, ora, (n, (L, 0.9 * L, 0.8 * L), (1, 1, 0), "uniform"))
