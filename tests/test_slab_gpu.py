"""Stride-1 windows straight from NCHW (tiles 35..46) at the edges where they can go wrong: one chunk of channels and a last one that is mostly padding,
slabs of one row group and of the most rows that fit, windows without padding and wider than they are high, one and two issuing warps, tiles in several
rounds, splits, tiles that end in the padding between images.  Integer operands: exact in any order, TF32 and fp16 alike."""
import os

import numpy as np
import pytest

from helpers import TF32_TOL, assert_parity, oracle_out, run_planned
from paper_1606_00094_b200 import workloads as wl

pytestmark = pytest.mark.gpu

F16 = 4
# (N,C,H,W,K,R,S,stride,pad,relu)
SHAPES = [
    (1, 3, 9, 11, 17, 3, 3, 1, 0, 1),            # one chunk of one MMA step, no padding
    (2, 70, 13, 13, 130, 3, 3, 1, 1, 0),         # a last chunk of six channels, images that end inside a tile
    (3, 33, 7, 9, 40, 2, 3, 1, 1, 1),            # R != S, one channel past a chunk
    (1, 40, 20, 60, 33, 7, 7, 1, 3, 1),          # slabs of 512 rows, one tap a stage
    (2, 96, 27, 27, 256, 5, 5, 1, 2, 1),         # three chunks: the sets of builders change places from tile to tile
    (31, 64, 24, 25, 90, 3, 3, 1, 1, 1),         # 159 tiles of positions: the second round of a persistent CTA
]


def _ints(shape, seed):
    N, C, H, W, K, R, S, *_ = shape
    return wl.integers(seed, (N, C, H, W)), wl.integers(seed + 1, (K, C, R, S)), wl.integers(seed + 2, (K,))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("tile", [35, 38, 41, 44, 46])           # 32, 80, 128, 192 and 256 channels
@pytest.mark.parametrize("math", [0, F16])
@pytest.mark.parametrize("split", [1, 3])
def test_slab_tiles_exact(shape, tile, math, split):
    x, w, b = _ints(shape, 7100)
    ref = oracle_out(shape, x, w, b)
    for bind in (False, True):
        got, desc = run_planned(shape, x, w, b, variant=2, math=math, tile_id=tile, split_k=split, bind=bind)
        assert "slab_128x" in desc and "workspace=0" in desc
        np.testing.assert_array_equal(got.astype(np.float64), ref, err_msg=desc)


# Windows by how their taps come to lie in stages (one, two, three or five taps of a row each) and how many stages a chunk and a row have: one stage a
# chunk is one issuing warp's, rows of one stage and of several wrap differently.  Several chunks, more tiles than SMs for the narrow tiles.
WINDOWS = [(2, 2, 1), (4, 4, 2), (1, 3, 0), (1, 2, 0), (1, 4, 0), (2, 1, 0), (3, 1, 0), (6, 6, 2), (9, 9, 4), (2, 10, 1)]


@pytest.mark.parametrize("R,S,pad", WINDOWS)
@pytest.mark.parametrize("math", [0, F16])
def test_windows_exact(R, S, pad, math):
    shape = (20, 70 if math == 0 else 130, 12, 11, 200, R, S, 1, pad, 1)
    x, w, b = _ints(shape, 7300)
    ref = oracle_out(shape, x, w, b)
    for tile in (35, 36, 37, 39, 40, 42, 43, 45):             # the widths that the shapes above leave out, and 32
        for split in (1, 2):
            got, desc = run_planned(shape, x, w, b, variant=2, math=math, tile_id=tile, split_k=split, bind=split == 1)
            assert "slab_128x" in desc
            np.testing.assert_array_equal(got.astype(np.float64), ref, err_msg=desc)


@pytest.mark.parametrize("tile,split", [(36, 1), (39, 2), (46, 1)])
@pytest.mark.parametrize("math", [0, F16])
def test_infinities_and_nan_stay_where_they_are(tile, split, math):
    """Positions that are computed and dropped, padding and the channels past the last one read as zeros beside them."""
    import torch
    from paper_1606_00094_b200 import binding as B
    shape = (3, 70, 9, 11, 50, 3, 3, 1, 1, 0)
    x, w, _ = _ints(shape, 7400)
    w[w == 0] = 1.0
    for value, at in ((np.inf, (0, 69, 0, 0)), (-np.inf, (1, 0, 8, 10)), (np.nan, (2, 33, 4, 0))):
        x[at] = value
    dx, dw = torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()
    want = torch.nn.functional.conv2d(dx.double(), dw.double(), padding=1).float()
    plan = B.ConvPlan(shape, variant=2, math=math, tile_id=tile, split_k=split)
    got = plan(dx, dw, None)
    plan.close()
    assert 0 < int((~torch.isfinite(want)).sum()) < want.numel() // 10
    assert torch.equal(torch.nan_to_num(got, nan=1e30), torch.nan_to_num(want, nan=1e30))


def test_filters_bound_again_between_calls():
    import torch
    from paper_1606_00094_b200 import binding as B
    shape = (20, 70, 13, 13, 130, 3, 3, 1, 1, 0)
    x, w, b = (torch.from_numpy(t).cuda() for t in _ints(shape, 7500))
    v = w.flip(0).contiguous()
    plan = B.ConvPlan(shape, variant=2, tile_id=39)
    refs = [torch.nn.functional.conv2d(x.double(), f.double(), b.double(), padding=1).float() for f in (w, v)]
    for bound, given, ref in ((w, w, 0), (v, v, 1), (None, w, 0), (None, v, 1), (w, w, 0)):
        if bound is not None:
            plan.bind_filters(bound)
        assert torch.equal(plan(x, given, b), refs[ref])
    w.copy_(v)                                                # the bound filters' values, bound again
    plan.bind_filters(w)
    assert torch.equal(plan(x, w, b), refs[1])
    plan.close()


@pytest.mark.parametrize("shape", [(2, 8, 12, 12, 16, 3, 3, 2, 1, 1), (2, 8, 12, 12, 16, 3, 3, 1, 3, 1), (1, 8, 8, 140, 16, 7, 7, 1, 3, 1)])
def test_what_the_slab_tiles_refuse(shape):
    """Strides, padding that is no part of the window, slabs of more than 512 rows."""
    from paper_1606_00094_b200 import binding as B
    with pytest.raises(B.BodaError) as e:
        B.ConvPlan(shape, variant=2, tile_id=38)
    assert e.value.status == B.BODA_ERR_UNSUPPORTED


@pytest.mark.parametrize("shape,slab", [((20, 256, 13, 13, 384, 3, 3, 1, 1, 1), True), ((128, 256, 13, 13, 384, 3, 3, 1, 1, 1), False),
                                        ((20, 256, 13, 13, 384, 3, 3, 2, 1, 1), False)])
def test_rule_takes_one_round_of_slabs(shape, slab):
    from paper_1606_00094_b200 import binding as B
    plan = B.ConvPlan(shape)
    try:
        assert ("slab_128x" in plan.describe()) == slab, plan.describe()
    finally:
        plan.close()


@pytest.mark.parametrize("shape", [(43, 191, 55, 57, 43, 3, 3, 1, 1, 1), (40, 163, 51, 52, 49, 3, 3, 1, 1, 1)])
def test_rule_leaves_many_chunks_of_fp16_to_the_pairs(shape):
    """Several rounds of narrow tiles: the slabs, twice the channels of a TF32 chunk each, take their builders longer than the tensor cores."""
    from paper_1606_00094_b200 import binding as B
    plan = B.ConvPlan(shape, math=F16)
    try:
        assert "pair_256x64" in plan.describe(), plan.describe()
    finally:
        plan.close()


# few tiles and several chunks: by rule with either storage, and in one call
@pytest.mark.parametrize("shape", [(1, 70, 5, 6, 33, 3, 3, 1, 1, 1), (1, 118, 16, 17, 86, 3, 3, 1, 1, 0)])
def test_few_tiles_by_rule_and_in_one_call(shape):
    import torch
    from paper_1606_00094_b200 import binding as B
    N, C, H, W, K, R, S, stride, pad, relu = shape
    x, w, b = wl.integers(15, (N, C, H, W)), wl.integers(16, (K, C, R, S)), wl.integers(17, (K,))
    ref = oracle_out(shape, x, w, b)
    for kw in (dict(math=F16), dict(variant=2)):
        got, desc = run_planned(shape, x, w, b, **kw)
        assert "slab_128x" in desc, desc
        np.testing.assert_array_equal(got.astype(np.float64), ref, err_msg=desc)
    y = B.conv_fwd(*(torch.from_numpy(a).cuda() for a in (x, w, b)), stride=stride, pad=pad, relu=bool(relu))
    np.testing.assert_array_equal(y.cpu().numpy().astype(np.float64), ref)


@pytest.mark.parametrize("tile,split", [(36, 1), (39, 2), (46, 1)])
def test_expired_wait_in_the_slab_kernel(tile, split):
    import torch
    from paper_1606_00094_b200 import binding as B
    shape = (3, 64, 13, 13, 200, 3, 3, 1, 1, 1)
    N, C, H, W, K, R, S, *_ = shape
    x, w, b = wl.half_normal(1, (N, C, H, W)), wl.normal(2, (K, C, R, S), 0, (2.0 / (C * R * S)) ** 0.5), wl.normal(3, (K,), 0, 0.01)
    dx, dw, db = (torch.from_numpy(t).cuda() for t in (x, w, b))
    assert B.boda_query_status() == 0
    os.environ["BODA_TEST_TX_MISMATCH"] = "1"
    os.environ["BODA_WAIT_LIMIT_CYCLES"] = "100000000"
    try:
        plan = B.ConvPlan(shape, variant=2, tile_id=tile, split_k=split)
    finally:
        del os.environ["BODA_TEST_TX_MISMATCH"]
        del os.environ["BODA_WAIT_LIMIT_CYCLES"]
    plan(dx, dw, db)
    torch.cuda.synchronize()
    assert B.boda_query_status() == B.BODA_ERR_DEVICE_TIMEOUT
    assert B.boda_query_status() == 0
    plan.close()
    got, desc = run_planned(shape, x, w, b, variant=2, tile_id=tile, split_k=split)
    assert_parity(got, oracle_out(shape, x, w, b), TF32_TOL, desc)
