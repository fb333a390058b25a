"""1x1 layers from NCHW in tiles of 64 and of 128 output points: images that end in any of a tile's boxes (those past the image are not loaded), one
round of tiles and several."""
import numpy as np
import pytest

from helpers import oracle_out, run_planned
from paper_1606_00094_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("points,shape", [
    (64, (2, 40, 2, 2, 50, 1, 1, 1, 0, 1)), (64, (2, 40, 6, 6, 50, 1, 1, 1, 0, 0)), (64, (1, 70, 10, 10, 130, 1, 1, 1, 0, 1)),
    (128, (160, 40, 2, 2, 50, 1, 1, 1, 0, 1)), (128, (150, 40, 6, 6, 50, 1, 1, 1, 0, 0)), (128, (90, 70, 10, 10, 60, 1, 1, 1, 0, 1)),
    (128, (150, 33, 14, 14, 70, 1, 1, 1, 0, 1)),
])
@pytest.mark.parametrize("tile", [20, 21])
def test_tiles_of_64_and_128_points_exact(points, shape, tile):
    N, C, H, W, K, *_ = shape
    x, w, b = wl.integers(5, (N, C, H, W)), wl.integers(6, (K, C, 1, 1)), wl.integers(7, (K,))
    got, desc = run_planned(shape, x, w, b, variant=1, tile_id=tile, split_k=1)
    assert f"points={points}" in desc, desc
    np.testing.assert_array_equal(got.astype(np.float64), oracle_out(shape, x, w, b), err_msg=desc)


# channel tiles that take turns with the CTAs (the grid of 148 is a multiple of 2 and 4, not of 3), the last of them ragged
@pytest.mark.parametrize("tile,shape", [
    (21, (160, 32, 6, 6, 139, 1, 1, 1, 0, 1)), (20, (90, 32, 6, 6, 196, 1, 1, 1, 0, 1)), (20, (160, 32, 6, 6, 139, 1, 1, 1, 0, 0)),
    (18, (240, 33, 7, 7, 139, 1, 1, 1, 0, 1)), (16, (160, 33, 7, 7, 230, 1, 1, 1, 0, 1)), (16, (160, 33, 7, 7, 139, 1, 1, 1, 0, 0)),
])
def test_channel_tiles_in_turn_exact(tile, shape):
    N, C, H, W, K, *_ = shape
    x, w, b = wl.integers(5, (N, C, H, W)), wl.integers(6, (K, C, 1, 1)), wl.integers(7, (K,))
    got, desc = run_planned(shape, x, w, b, variant=1, tile_id=tile, split_k=1)
    np.testing.assert_array_equal(got.astype(np.float64), oracle_out(shape, x, w, b), err_msg=desc)


@pytest.mark.parametrize("shape", [(6, 336, 56, 56, 22, 1, 1, 1, 0, 1), (23, 362, 28, 28, 20, 1, 1, 1, 0, 1)])
def test_a_few_tiles_of_a_second_round_do_not_change_the_kernel(shape):
    """150 and 161 tiles on 148 SMs."""
    from paper_1606_00094_b200 import binding as B
    plan = B.ConvPlan(shape)
    try:
        assert "k1nchw_128x64" in plan.describe(), plan.describe()
    finally:
        plan.close()
