"""Sort and neighbour bins where the scan over blocks of cells has one tile of 4096
blocks (64^3 cells without a split by material: exactly 4096) and where it has more
(the same sort with water apart, two scenes, 128^3 codes of a 70^3 grid). The same
check and tolerance as the smaller grids'."""
import pytest

import test_gpu_sort

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,counts", [(64, (640,)), (64, (640, 33)), (70, (500,)), (70, (200, 0, 300))])
def test_tiles(n, counts):
    test_gpu_sort.test_neighbour_sums_and_order(n, counts)
