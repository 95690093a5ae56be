"""Dual clipping at every number of warps a channel can get, at value counts off the vector width, and with more values per
channel than shared memory holds."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,D,iters", [
    (37, 9, 20), (131, 300, 30), (1003, 640, 20), (257, 1200, 20), (66, 2500, 20), (6001, 600, 5), (51300, 8, 5),
])
def test_dual_clip_sizes_match_oracle(n, D, iters):
    parity.check_dual_clip(n, D, 4, seed=n + D, iters=iters)


@pytest.mark.parametrize("n,D,iters,strided", [
    (131, 200, 40, False), (131, 300, 40, True), (1003, 640, 40, True), (257, 1200, 40, False), (66, 2500, 40, True),
])
def test_sorted_values_match_oracle_at_every_number_of_warps(n, D, iters, strided):
    """16, 8, 4, 2 and 1 warps per channel (28 per SM over all channels); 32 steps and more at 4 bits take the sorted values."""
    parity.check_dual_clip(n, D, 4, seed=n + D, iters=iters, strided=strided)
