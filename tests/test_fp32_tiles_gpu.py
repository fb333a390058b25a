"""FP32 (DIRECT) kernels at the sizes where they can go wrong: GEMM-blocked tiles with the reduction split over a cluster, and the
tiles that run over a staged copy of the input with their work cut into equal pieces.  Integer-valued operands make every
partial sum exact, so any order of summation must give the oracle's bits."""
import numpy as np
import pytest

from helpers import oracle_out, run_planned
from paper_1606_00094_b200 import workloads as wl

pytestmark = pytest.mark.gpu

# (N,C,H,W,K,R,S,stride,pad,relu)
SHAPES = [
    (1, 1, 5, 5, 1, 1, 1, 1, 0, 0),              # one reduction index, one channel, far less than any tile
    (2, 5, 9, 11, 33, 3, 3, 1, 1, 1),            # odd reduction length (no 8-byte filter copies), a channel past a tile
    (3, 36, 13, 13, 97, 3, 3, 1, 1, 1),          # a chunk and one 4-channel group, points one past several tiles
    (1, 34, 12, 13, 49, 5, 5, 2, 2, 1),          # channels not a multiple of 4, stride 2
    (2, 4, 23, 20, 50, 6, 6, 1, 3, 1),           # more taps than the bounds mask holds
    (1, 3, 40, 37, 130, 11, 11, 4, 0, 0),        # large window, stride 4
    (5, 64, 7, 7, 128, 2, 4, 1, 1, 1),           # R != S
]


def _ints(shape, seed):
    N, C, H, W, K, R, S, *_ = shape
    return wl.integers(seed, (N, C, H, W)), wl.integers(seed + 1, (K, C, R, S)), wl.integers(seed + 2, (K,))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("tile", [0, 1, 2, 3, 4, 5, 6, 7, 8, 16, 17])
def test_gemm_tiles_and_splits_exact(shape, tile):
    x, w, b = _ints(shape, 9100)
    ref = oracle_out(shape, x, w, b)
    for split in (1, 3, 8):
        got, desc = run_planned(shape, x, w, b, variant=0, math=1, tile_id=tile, split_k=split)
        assert f"id {tile}" in desc
        np.testing.assert_array_equal(got.astype(np.float64), ref, err_msg=desc)


@pytest.mark.parametrize("shape", SHAPES + [(60, 8, 24, 24, 40, 1, 1, 1, 0, 1),        # 270 tiles of 128 points: nearly two rounds of the SMs, cut into equal pieces
                                            (148, 4, 16, 16, 8, 1, 1, 1, 0, 1),        # exactly two rounds, nothing cut
                                            (79, 4, 32, 32, 8, 1, 1, 1, 0, 1)])        # whole rounds first, then the cut remainder
@pytest.mark.parametrize("tile", [18, 19, 20, 21, 22])
@pytest.mark.parametrize("bind", [False, True])
def test_staged_tiles_exact(shape, tile, bind):
    x, w, b = _ints(shape, 9200)
    got, desc = run_planned(shape, x, w, b, variant=0, math=1, tile_id=tile, bind=bind)
    assert "direct_nhwc" in desc
    np.testing.assert_array_equal(got.astype(np.float64), oracle_out(shape, x, w, b), err_msg=desc)


def test_filters_off_an_8_byte_boundary():
    import torch
    from paper_1606_00094_b200 import binding as B
    shape = (2, 4, 9, 11, 33, 3, 3, 1, 1, 1)                 # even reduction length: only the address rules the pair copies out
    x, w, b = _ints(shape, 9300)
    store = torch.zeros(w.size + 1, device="cuda")
    off = store[1:].view(w.shape)
    off.copy_(torch.from_numpy(w))
    assert off.data_ptr() % 8 == 4
    for tile in (2, 7, 16, 18):
        plan = B.ConvPlan(shape, variant=0, math=1, tile_id=tile)
        got = plan(torch.from_numpy(x).cuda(), off, torch.from_numpy(b).cuda()).cpu().numpy()
        np.testing.assert_array_equal(got.astype(np.float64), oracle_out(shape, x, w, b))


@pytest.mark.parametrize("tile,split", [(2, 8), (7, 3), (18, 0), (21, 0)])
def test_every_run_gives_the_same_bits(tile, split):
    shape = (7, 50, 14, 15, 70, 3, 3, 1, 1, 1)
    N, C, H, W, K, R, S, *_ = shape
    x, w, b = wl.half_normal(1, (N, C, H, W)), wl.normal(2, (K, C, R, S), 0.0, 0.07), wl.normal(3, (K,), 0.0, 0.01)
    runs = [run_planned(shape, x, w, b, variant=0, math=1, tile_id=tile, split_k=split)[0] for _ in range(2)]
    assert np.array_equal(runs[0], runs[1])


@pytest.mark.parametrize("shape,name", [((20, 256, 13, 13, 384, 3, 3, 1, 1, 1), "direct_nhwc_x3_128x"), ((3, 328, 11, 13, 9, 11, 11, 4, 0, 1), "direct_nhwc_128x")])
def test_workspace_limit_keeps_fp32_plans_off_the_staged_tiles(shape, name):
    from paper_1606_00094_b200 import binding as B
    assert name in B.ConvPlan(shape, math=1).describe()
    plan = B.ConvPlan(shape, math=1, max_workspace=4096)
    assert "workspace=0" in plan.describe() and "direct_nhwc" not in plan.describe()
    with pytest.raises(B.BodaError) as e:
        B.ConvPlan(shape, math=1, variant=0, tile_id=18, max_workspace=4096)
    assert e.value.status == B.BODA_ERR_NOMEM


def test_tuning_an_fp32_layer_with_a_forced_split_times_its_tiles(tmp_path, monkeypatch):
    from paper_1606_00094_b200 import binding as B
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("BODA_TUNE_CACHE", str(cache))
    plan = B.ConvPlan((3, 36, 13, 13, 97, 3, 3, 1, 1, 1), math=B.BODA_MATH_FP32, tune=1, split_k=3)
    try:
        # (nothing is written down where nothing was timed)
        assert cache.exists() and len(cache.read_text().strip().splitlines()) == 1
        assert "split_k=3" in plan.describe() or "split_k=1" in plan.describe()      # 1: a tile that does not split was faster
    finally:
        plan.close()
