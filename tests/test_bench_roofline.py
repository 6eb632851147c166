"""The benchmark states a roofline only for the kernel that its operation count is of."""
import pytest

import bench
from paper_1912_12453_gb300 import chns


@pytest.mark.parametrize("schedule", range(len(chns.JACVEC_VARIANTS)))
def test_flop_count_belongs_to_the_schedule(schedule):
    pair = "two Gauss points per lane" in chns.JACVEC_VARIANTS[schedule]
    assert (bench.jv_flop_per_leaf(3, schedule) is not None) == pair
