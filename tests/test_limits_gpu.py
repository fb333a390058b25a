"""Limits on workspace and forced splits: which calls are refused, and in which arithmetic the others run.  Kernels that need no workspace do not change
either: where every kernel that stages its input is ruled out, a window layer runs in FP32 by rule and is refused as a named variant."""
import pytest

pytestmark = pytest.mark.gpu

K1, TC = 1, 2
F16 = 4


def _plan(shape, **kw):
    from paper_1606_00094_b200 import binding as B
    plan = B.ConvPlan(shape, **kw)
    desc = plan.describe()
    plan.close()
    return desc


# many tiles of positions and few; windows of 9 and 21 taps, more than 1536 indices (no gather kernel)
WINDOWS = [(20, 256, 13, 13, 384, 3, 3, 1, 1, 1), (1, 256, 13, 13, 384, 3, 3, 1, 1, 1), (22, 80, 3, 20, 338, 3, 7, 1, 2, 1)]


@pytest.mark.parametrize("shape", WINDOWS)
@pytest.mark.parametrize("tune", [0, 1])
def test_a_window_layer_under_a_tight_limit(shape, tune):
    from paper_1606_00094_b200 import binding as B
    assert "math=tf32" in _plan(shape)
    assert "math=fp32" in _plan(shape, max_workspace=1024, tune=tune)
    assert "math=fp32" in _plan(shape, max_workspace=1024, split_k=1)
    with pytest.raises(B.BodaError) as e:
        B.ConvPlan(shape, variant=TC, max_workspace=1024, tune=tune)
    assert e.value.status == B.BODA_ERR_NOMEM


def test_a_remembered_choice_under_a_tight_limit(tmp_path, monkeypatch):
    """A slab tile that tuning found without a limit is not taken from the file where the limit rules the others out."""
    from paper_1606_00094_b200 import binding as B
    monkeypatch.setenv("BODA_TUNE_CACHE", str(tmp_path / "tune.txt"))
    shape = (1, 200, 16, 17, 86, 3, 3, 1, 1, 1)               # 1800 indices: no gather kernel
    assert "slab_128x" in _plan(shape, variant=TC, tune=1)
    assert "slab_128x" in _plan(shape, variant=TC, tune=1, max_workspace=1 << 20)
    with pytest.raises(B.BodaError) as e:
        B.ConvPlan(shape, variant=TC, max_workspace=1024, tune=1)
    assert e.value.status == B.BODA_ERR_NOMEM


@pytest.mark.parametrize("shape", WINDOWS)
def test_the_same_with_fp16_storage(shape):
    from paper_1606_00094_b200 import binding as B
    assert "math=f16" in _plan(shape, math=F16)
    assert "math=fp32" in _plan(shape, math=F16, max_workspace=1024)
    with pytest.raises(B.BodaError) as e:
        B.ConvPlan(shape, math=F16, variant=TC, max_workspace=1024)
    assert e.value.status == B.BODA_ERR_NOMEM


def test_a_forced_split_of_a_1x1_layer():
    """The gather kernel has no split: under a limit that staging does not fit, the kernel that reads NCHW by TMA runs, and is not refused."""
    shape = (600, 64, 2, 2, 64, 1, 1, 1, 0, 1)
    assert "gconv" in _plan(shape, variant=K1, max_workspace=1024)
    assert "k1nchw" in _plan(shape, variant=K1, split_k=2, max_workspace=1024)


@pytest.mark.parametrize("shape,split", [((38, 150, 14, 14, 184, 1, 1, 1, 0, 1), 3), ((23, 40, 34, 40, 157, 1, 1, 1, 0, 1), 2)])
def test_a_forced_split_rounds_its_operands(shape, split):
    """Layers whose operands are rounded to TF32 under a forced split are not handed to the kernel that cuts them off."""
    assert "tile=igemm" in _plan(shape, variant=K1, split_k=split)
