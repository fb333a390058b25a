"""CTA-pair tiles (ids 26..30) at the edges where they can go wrong: second CTA of a tile without points, ragged channels, an odd
number of reduction chunks (the last stage of a tile is half full), chunks whose padding steps are skipped, more tiles than
pairs (both accumulators in turn), staged output through tensor stores.  Integer operands: exact in any order."""
import numpy as np
import pytest

from helpers import FP32_TOL, assert_parity, oracle_out, run_planned
from paper_1606_00094_b200 import workloads as wl

pytestmark = pytest.mark.gpu

# (N,C,H,W,K,R,S,stride,pad,relu)
SHAPES = [
    (1, 32, 9, 9, 33, 1, 1, 1, 0, 0),            # one reduction chunk, 81 points: the second CTA has none
    (2, 8, 13, 13, 64, 3, 3, 1, 1, 1),           # one MMA step per chunk
    (3, 72, 13, 13, 130, 3, 3, 1, 1, 1),         # three chunks of 32, last one a quarter full; 507 points
    (1, 96, 27, 27, 257, 5, 5, 1, 2, 1),         # a channel past the widest tile; fp16: last chunk half full
    (5, 40, 21, 20, 60, 3, 3, 2, 1, 0),          # stride 2
    (11, 64, 43, 43, 100, 1, 1, 1, 0, 1),        # 80 tiles of 256 points: more than the pairs
    (24, 16, 28, 28, 300, 3, 3, 1, 1, 1),        # every width has several rounds
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("tile", [26, 27, 28, 29, 30])
@pytest.mark.parametrize("math", [0, 4])
def test_pair_tiles_exact(shape, tile, math):
    N, C, H, W, K, R, S, *_ = shape
    x, w, b = wl.integers(9500, (N, C, H, W)), wl.integers(9501, (K, C, R, S)), wl.integers(9502, (K,))
    ref = oracle_out(shape, x, w, b)
    for bind in (False, True):
        got, desc = run_planned(shape, x, w, b, variant=1 if R * S == 1 else 2, math=math, tile_id=tile, s2d=0, bind=bind)
        assert "pair_256" in desc
        np.testing.assert_array_equal(got.astype(np.float64), ref, err_msg=desc)


@pytest.mark.parametrize("tile", [26, 28, 30])
@pytest.mark.parametrize("consumer", [-1, 6])            # an im2col reader (tensor stores) and a halo reader (padded rows)
def test_pair_tiles_in_a_chain(tile, consumer):
    import torch
    from oracle import conv_oracle as orc
    from paper_1606_00094_b200.stack import ConvStack
    ops = [wl.StackOp("conv", wl.ConvShape(7, 40, 15, 17, 96, 3, 3, 1, 1)), wl.StackOp("conv", wl.ConvShape(7, 96, 15, 17, 70, 3, 3, 1, 1)), wl.StackOp("pool")]
    # 40*9 products of at most 4 each stay below 2^11, so the first layer's outputs are exact TF32 values; the second layer's
    # are integers below 2^24 that its staged output rounds to TF32 (nearest, ties away) on the way to the pool
    x = wl.integers(9600, (7, 40, 15, 17), -2, 2)
    params = [(wl.integers(9601 + i, (o.shape.K, o.shape.C, 3, 3), -2, 2), wl.integers(9611 + i, (o.shape.K,))) for i, o in enumerate(ops[:2])]
    stack = ConvStack(ops, params, per_op=[{"variant": 2, "tile_id": tile}, {"variant": 2, "tile_id": consumer} if consumer >= 0 else {}, {}])
    got = stack.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    descs = stack.describe()
    stack.close()
    assert "pair_256" in descs[0] and "out=staged" in descs[0]
    a = orc.conv_fwd(x, *params[0], stride=1, pad=1, relu=True)
    assert np.abs(a).max() < 2048
    a = orc.conv_fwd(a.astype(np.float32), *params[1], stride=1, pad=1, relu=True).astype(np.float32)
    a = ((a.view(np.int32) + 0x1000) & ~0x1FFF).view(np.float32)
    np.testing.assert_array_equal(got.astype(np.float64), orc.maxpool_fwd(a), err_msg=str(descs))


def _as_tf32(a):
    """The value the staging kernel stores: nearest TF32, ties away."""
    return ((a.view(np.int32) + 0x1000) & ~0x1FFF).view(np.float32)


def _accumulation_error(shape, math, **plan):
    """Real-valued operands; the oracle is fed what the staging kernel stores, which leaves fp32 accumulation as the only difference."""
    N, C, H, W, K, R, S, *_ = shape
    x, w, b = wl.half_normal(9700, (N, C, H, W)), wl.normal(9701, (K, C, R, S), 0.0, (2.0 / (C * R * S)) ** 0.5), wl.normal(9702, (K,), 0.0, 0.01)
    staged = [a.astype(np.float16).astype(np.float32) if math == 4 else _as_tf32(a) for a in (x, w)]
    got, desc = run_planned(shape, x, w, b, math=math, **plan)
    return assert_parity(got, oracle_out(shape, *staged, b), FP32_TOL, desc), desc


@pytest.mark.parametrize("shape", [(2, 512, 13, 13, 100, 3, 3, 1, 1, 1), (3, 1024, 14, 14, 160, 1, 1, 1, 0, 0), (2, 70, 13, 13, 70, 5, 5, 1, 2, 0)])
@pytest.mark.parametrize("tile", [26, 28, 30])
@pytest.mark.parametrize("math", [0, 4])
def test_real_valued_sums(shape, tile, math):
    _, desc = _accumulation_error(shape, math, variant=1 if shape[5] * shape[6] == 1 else 2, tile_id=tile, s2d=0)
    assert "pair_256" in desc


def test_longest_sums_by_rule():
    """Layers of several rounds of tiles, which suit the pairs, with reductions of 7100 and 11650: the FP32 bar on staged operands
    holds for what the rule picks."""
    _accumulation_error((47, 284, 24, 24, 84, 5, 5, 1, 2, 0), 4)
    _accumulation_error((11, 466, 28, 28, 59, 5, 5, 1, 2, 0), 4)
    _accumulation_error((11, 466, 28, 28, 59, 5, 5, 1, 2, 0), 0)


@pytest.mark.parametrize("tile", [26, 28, 30])
@pytest.mark.parametrize("shape", [(3, 8, 31, 29, 70, 5, 5, 2, 2, 1), (2, 3, 67, 67, 100, 11, 11, 4, 0, 1), (2, 20, 22, 23, 33, 3, 3, 3, 1, 0)])
def test_pair_tiles_on_a_space_to_depth_view_exact(shape, tile):
    N, C, H, W, K, R, S, *_ = shape
    x, w, b = wl.integers(9800, (N, C, H, W)), wl.integers(9801, (K, C, R, S)), wl.integers(9802, (K,))
    for bind in (False, True):
        got, desc = run_planned(shape, x, w, b, variant=2, tile_id=tile, s2d=1, bind=bind)
        assert "pair_256" in desc and "s2d" in desc
        np.testing.assert_array_equal(got.astype(np.float64), oracle_out(shape, x, w, b), err_msg=desc)


@pytest.mark.parametrize("shape", [(14, 3, 150, 150, 48, 7, 7, 2, 0, 1), (33, 3, 215, 215, 48, 5, 5, 2, 2, 1),       # strided first layers
                                   (18, 16, 34, 34, 106, 3, 3, 2, 1, 1),                                             # 16 channels, stride 2
                                   (227, 75, 13, 13, 356, 1, 1, 1, 0, 1)])                                           # three steps a tile
def test_rule_leaves_these_to_the_gather_kernel(shape):
    from paper_1606_00094_b200 import binding as B
    plan = B.ConvPlan(shape)
    try:
        assert "gconv" in plan.describe()
    finally:
        plan.close()


def test_rule_leaves_one_round_of_halo_tiles_alone():
    """11x11 with stride 4: 139 halo tiles of 512 positions, where pairs would begin a fourth round."""
    from paper_1606_00094_b200 import binding as B
    plan = B.ConvPlan((35, 3, 171, 171, 32, 11, 11, 4, 5, 1))
    try:
        assert "halo_512x64" in plan.describe(), plan.describe()
    finally:
        plan.close()
