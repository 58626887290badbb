"""Mixed batches whose row groups are the fewest the batch can have (every group gets the same number of blocks) and one more than
that (blocks in proportion), against the CPU oracle: greedy, sampling, filtered sampling."""
import pytest

import test_gpu_odd_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("V,counts", [(9000, (20, 15, 0, 0)), (9000, (24, 24, 0, 0)), (20000, (32, 32, 32, 32)), (70008, (40, 0, 0, 0)),
                                      (20000, (33, 31, 0, 0)), (1000, (7, 0, 0, 0)), (9000, (130, 0, 0, 0)), (705, (8, 8, 8, 8))])
def test_groups_of_about_the_same_size(V, counts, pad):
    test_gpu_odd_rows.test_groups_of_very_different_size(V, counts, pad)
