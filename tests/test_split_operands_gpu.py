"""Tiles that multiply operands split into three bf16 parts on the tensor cores (31..34 in the error-compensated mode, 23..26 of the FP32
kernels) at the edges where they can go wrong: one chunk, chunks whose padding steps are skipped, ragged channels and points, periods that
do not divide the reduction, more tiles than SMs, splits.  Integer operands: exact in any order."""
import os

import numpy as np
import pytest

from helpers import FP32_TOL, assert_parity, oracle_out, run_planned
from paper_1606_00094_b200 import workloads as wl

pytestmark = pytest.mark.gpu

# (N,C,H,W,K,R,S,stride,pad,relu)
SHAPES = [
    (1, 5, 7, 9, 3, 1, 1, 1, 0, 0),              # one chunk of one MMA step, less than any tile
    (2, 70, 13, 13, 81, 3, 3, 1, 1, 1),          # second chunk one step long, a channel past a tile
    (3, 64, 12, 13, 130, 5, 5, 2, 2, 1),         # stride 2, 25 chunks: an odd number, so the last period is short
    (1, 200, 9, 11, 97, 2, 4, 1, 1, 0),          # R != S
    (40, 16, 23, 23, 65, 3, 3, 1, 1, 1),         # 166 tiles of points: the second round of a persistent CTA
]


def _ints(shape, seed):
    N, C, H, W, K, R, S, *_ = shape
    return wl.integers(seed, (N, C, H, W)), wl.integers(seed + 1, (K, C, R, S)), wl.integers(seed + 2, (K,))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("tile", [0, 1, 2, 3])
@pytest.mark.parametrize("split", [1, 3, 8])
def test_split_tiles_exact(shape, tile, split):
    x, w, b = _ints(shape, 9800)
    ref = oracle_out(shape, x, w, b)
    got, desc = run_planned(shape, x, w, b, variant=1 if shape[5] * shape[6] == 1 else 2, math=3, tile_id=31 + tile, split_k=split, bind=True)
    assert "split_128x" in desc
    np.testing.assert_array_equal(got.astype(np.float64), ref, err_msg=desc)
    got, desc = run_planned(shape, x, w, b, variant=0, math=1, tile_id=23 + tile, split_k=split)
    assert "direct_nhwc_x3" in desc
    np.testing.assert_array_equal(got.astype(np.float64), ref, err_msg=desc)


def test_operands_keep_all_their_bits():
    """A window that picks one input out: the sum has one product, so nothing but the operands' parts can lose anything."""
    rng = np.random.default_rng(3)
    x = rng.standard_normal((2, 33, 9, 9)).astype(np.float32) * np.exp2(rng.integers(-60, 60, (2, 33, 9, 9))).astype(np.float32)
    w = np.zeros((33, 33, 3, 3), np.float32)
    w[np.arange(33), np.arange(33), 1, 1] = 1.0
    got, _ = run_planned((2, 33, 9, 9, 33, 3, 3, 1, 1, 0), x, w, None, variant=0, math=1, tile_id=24)
    np.testing.assert_array_equal(got, x)
    got, _ = run_planned((2, 33, 9, 9, 33, 3, 3, 1, 1, 0), np.ones_like(x), w * x[0, :, 4, 4][:, None, None, None], None, variant=0, math=1, tile_id=24)
    np.testing.assert_array_equal(got, np.broadcast_to(x[0, :, 4, 4][None, :, None, None], got.shape))


@pytest.mark.parametrize("tile", [24, 26])
def test_small_and_large_operands_keep_all_their_bits(tile):
    """The same for operands from 2^-124, whose last bit is 2^-147, to 2^127."""
    rng = np.random.default_rng(4)
    size = (2, 33, 9, 9)
    x = (rng.uniform(1, 2, size) * rng.choice([-1, 1], size)).astype(np.float32)
    x = np.ldexp(x, rng.choice([-124, -123, -120, -116, -111, -109, -80, 0, 100, 126, 127], size)).astype(np.float32)
    w = np.zeros((33, 33, 3, 3), np.float32)
    w[np.arange(33), np.arange(33), 1, 1] = 1.0
    shape = (2, 33, 9, 9, 33, 3, 3, 1, 1, 0)
    x = np.where(np.arange(33)[None, :, None, None] == 5, np.float32(np.finfo(np.float32).max), x)
    got, desc = run_planned(shape, x, w, None, variant=0, math=1, tile_id=tile)
    np.testing.assert_array_equal(got, x, err_msg=desc)
    f = x[0, :, 4, 4]
    got, desc = run_planned(shape, np.ones_like(x), w * f[:, None, None, None], None, variant=0, math=1, tile_id=tile)
    np.testing.assert_array_equal(got, np.broadcast_to(f[None, :, None, None], got.shape), err_msg=desc)


@pytest.mark.parametrize("kw", [dict(variant=0, math=1, tile_id=t) for t in (23, 24, 25, 26)] + [dict(variant=2, math=3, tile_id=t) for t in (32, 34)])
@pytest.mark.parametrize("scale", [-118, 110])
def test_layers_of_small_and_large_operands(scale, kw):
    """No further off than with operands around one (the bound of test_no_further_off_than_fp32_arithmetic)."""
    from oracle import conv_oracle as orc
    shape = (2, 256, 13, 13, 96, 3, 3, 1, 1, 0)
    x, w = np.ldexp(wl.half_normal(1, shape[:1] + shape[1:4]), scale).astype(np.float32), wl.normal(2, (96, 256, 3, 3), 0, (2.0 / 2304) ** 0.5)
    got, desc = run_planned(shape, x, w, None, **kw)
    assert orc.rel_l2(np.ldexp(got.astype(np.float64), -scale), np.ldexp(oracle_out(shape, x, w, None), -scale)) <= 1.3e-7 + 2.0 ** -24 * (1.0 + np.sqrt(2304 / 256.0)), desc


@pytest.mark.parametrize("shape", [(2, 256, 13, 13, 96, 3, 3, 1, 1, 1), (1, 900, 6, 6, 64, 5, 5, 1, 2, 0)])
@pytest.mark.parametrize("tile", [23, 24, 25, 26])
def test_no_further_off_than_fp32_arithmetic(shape, tile):
    """A sum of n terms in FP32 is off by about 2^-24 * sqrt(n / 4) of itself on the FP32 tiles (two running sums, errors of random sign):
    8e-7 for 2304 terms.  Here an accumulator takes two chunks (8 MMAs at 1.6e-8: 1.3e-7), whatever n is, and n / 128 of them are added."""
    from oracle import conv_oracle as orc
    N, C, H, W, K, R, S, *_ = shape
    x, w, b = wl.half_normal(1, (N, C, H, W)), wl.normal(2, (K, C, R, S), 0, (2.0 / (C * R * S)) ** 0.5), wl.normal(3, (K,), 0, 0.01)
    ref = oracle_out(shape, x, w, b)
    runs = [run_planned(shape, x, w, b, variant=0, math=1, tile_id=tile)[0] for _ in range(2)]
    assert np.array_equal(runs[0], runs[1])
    assert orc.rel_l2(runs[0], ref) <= 1.3e-7 + 2.0 ** -24 * (1.0 + np.sqrt(C * R * S / 256.0))


@pytest.mark.parametrize("bits", [0x3f80ffff, 0x3f807f40])
@pytest.mark.parametrize("tile", [23, 24, 25, 26])
def test_products_of_the_worst_operands(bits, tile):
    """All operands the value whose parts leave most out: with parts cut off, 0x3f80ffff (ml + lm is 2^-21 of the product); with parts rounded to
    nearest, 0x3f807f40 (2^-24).  64 equal products: sums of hh and of the mixed ones are exact, or off by 2^-24 once; one more
    rounding where they meet."""
    from oracle import conv_oracle as orc
    value = np.uint32(bits).view(np.float32)
    x, w = np.full((1, 64, 5, 5), value, np.float32), np.full((70, 64, 1, 1), value, np.float32)
    shape = (1, 64, 5, 5, 70, 1, 1, 1, 0, 0)
    got, desc = run_planned(shape, x, w, None, variant=0, math=1, tile_id=tile)
    assert orc.rel_l2(got, oracle_out(shape, x, w, None)) <= 3 * 2.0 ** -24, desc


def test_an_infinity_times_the_smallest_values_is_one():
    for value in (1e-45, -1e-42, 9e-41, 0.0):
        x, w = np.full((1, 1, 4, 4), np.inf, np.float32), np.full((1, 1, 1, 1), value, np.float32)
        for args in ((x, w), (np.full_like(x, value), np.full_like(w, np.inf))):
            import torch
            from paper_1606_00094_b200 import binding as B
            plan = B.ConvPlan((1, 1, 4, 4, 1, 1, 1, 1, 0, 0), math=1, variant=0, tile_id=24)
            got = plan(*[torch.from_numpy(t).cuda() for t in args]).cpu().numpy()
            plan.close()
            assert np.isnan(got).all() if value == 0 else np.array_equal(got, np.full_like(got, np.copysign(np.inf, value)))


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 3.4e38])
def test_infinities_and_nans_come_out_as_from_fp32_arithmetic(bad):
    import torch
    from paper_1606_00094_b200 import binding as B
    shape = (1, 40, 9, 9, 70, 3, 3, 1, 1, 0)
    x, w, b = wl.normal(5, (1, 40, 9, 9), 0, 1), wl.normal(6, (70, 40, 3, 3), 0, 0.1), wl.normal(7, (70,), 0, 0.01)
    x[0, 11, 4, 4] = bad
    with np.errstate(all="ignore"):
        want = oracle_out(shape, x, w, b).astype(np.float32)
    args = [torch.from_numpy(t).cuda() for t in (x, w, b)]
    for tile in (18, 23, 26):
        got = B.ConvPlan(shape, math=1, variant=0, tile_id=tile)(*args).cpu().numpy()
        assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isposinf(got), np.isposinf(want)), tile
        assert np.array_equal(np.isneginf(got), np.isneginf(want)), tile
        ok = np.isfinite(want)
        assert np.linalg.norm((got[ok] - want[ok]).astype(np.float64) / 1e30) <= FP32_TOL * np.linalg.norm(want[ok].astype(np.float64) / 1e30)


def test_rule_and_workspace():
    from paper_1606_00094_b200 import binding as B
    shape = (20, 256, 13, 13, 384, 3, 3, 1, 1, 1)
    plan = B.ConvPlan(shape, math=B.BODA_MATH_FP32)
    assert "direct_nhwc_x3" in plan.describe() and B.boda_conv_plan_kernels_per_call(plan.handle) == 2
    x, w, b = _ints(shape, 9810)
    ref = oracle_out(shape, x, w, b)
    for variant, math, tile in ((-1, 1, -1), (0, 0, -1), (-1, 3, -1)):
        got, desc = run_planned(shape, x, w, b, variant=variant, math=math, tile_id=tile)
        assert "x3" in desc
        np.testing.assert_array_equal(got.astype(np.float64), ref, err_msg=desc)
    with pytest.raises(B.BodaError) as e:
        B.ConvPlan(shape, math=1, variant=0, tile_id=24, max_workspace=4096)
    assert e.value.status == B.BODA_ERR_NOMEM
    for tile in (31, 34):                         # tiles of the error-compensated mode only
        with pytest.raises(B.BodaError):
            B.ConvPlan(shape, math=2, variant=2, tile_id=tile)


def test_workspace_stays_in_proportion_to_the_tensors():
    """16 channels: the parts of a chunk of 64 are six times the input.  Picked by rule or by the tuner, they may take four times input and
    output together; a caller who names a limit or a tile has what was asked for."""
    from paper_1606_00094_b200 import binding as B
    shape = (64, 16, 224, 224, 96, 11, 11, 4, 2, 1)
    points, tensors = 64 * 224 * 224, 4 * (64 * 16 * 224 * 224 + 64 * 96 * 55 * 55)
    need = points * 384
    assert 256 << 20 < 4 * tensors < need
    for kw in (dict(math=1), dict(math=3), dict(math=1, tune=1)):
        plan = B.ConvPlan(shape, **kw)
        assert "x3_128" not in plan.describe() and "split_128" not in plan.describe(), plan.describe()
        plan.close()
    for kw in (dict(math=1, max_workspace=2 * need), dict(math=1, variant=0, tile_id=25), dict(math=3, variant=2, tile_id=33)):
        plan = B.ConvPlan(shape, **kw)
        assert B.boda_conv_plan_workspace_bytes(plan.handle) == need, plan.describe()
        plan.close()


@pytest.mark.parametrize("tile,split", [(31, 1), (34, 1), (33, 3)])
def test_expired_wait(tile, split):
    import torch
    from paper_1606_00094_b200 import binding as B
    shape = (3, 64, 13, 13, 200, 3, 3, 1, 1, 1)
    x, w, b = _ints(shape, 9820)
    args = [torch.from_numpy(t).cuda() for t in (x, w, b)]
    os.environ["BODA_TEST_TX_MISMATCH"] = "1"
    os.environ["BODA_WAIT_LIMIT_CYCLES"] = "100000000"
    try:
        plan = B.ConvPlan(shape, variant=2, math=3, tile_id=tile, split_k=split)
    finally:
        del os.environ["BODA_TEST_TX_MISMATCH"]
        del os.environ["BODA_WAIT_LIMIT_CYCLES"]
    plan(*args)
    torch.cuda.synchronize()
    assert B.boda_query_status() == B.BODA_ERR_DEVICE_TIMEOUT
    assert B.boda_query_status() == 0
    plan.close()
    got, desc = run_planned(shape, x, w, b, variant=2, math=3, tile_id=tile, split_k=split)
    assert_parity(got, oracle_out(shape, x, w, b), 0.0, desc)


# layers around the line between the tiles of split operands and the others, measured times (us) split operands / the other kernel
KEEP_OTHER = [
    ((31, 79, 113, 116, 1, 3, 3, 1, 1, 0), 1),        # 562 / 363: one filter, a staged copy that L2 does not hold
    ((22, 16, 82, 83, 17, 3, 3, 1, 1, 0), 1),         # 70 / 47: three quarters of a chunk are padding
    ((36, 2, 105, 107, 119, 2, 2, 4, 0, 0), 3),       # 53 / 34
    ((48, 5, 113, 116, 130, 1, 1, 2, 0, 0), 3),       # 123 / 87
]
TAKE_SPLIT = [((20, 256, 13, 13, 384, 3, 3, 1, 1, 1), 1), ((20, 64, 56, 56, 128, 3, 3, 1, 1, 1), 1), ((5, 256, 13, 13, 384, 3, 3, 1, 1, 1), 3)]


@pytest.mark.parametrize("shape,math", KEEP_OTHER + TAKE_SPLIT)
def test_line_between_split_operands_and_the_other_kernels(shape, math):
    from paper_1606_00094_b200 import binding as B
    plan = B.ConvPlan(shape, math=math)
    desc = plan.describe()
    plan.close()
    assert ("direct_nhwc_x3_128x" in desc or "split_128x" in desc) == ((shape, math) in TAKE_SPLIT), desc
