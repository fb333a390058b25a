"""Operand staging (input and filters in one launch) at its edges, seen through the layers that read it: integer-valued operands
must come out exactly whatever the staging does with padding, ragged tiles and window sizes."""
import numpy as np
import pytest

from helpers import oracle_out, run_planned
from paper_1606_00094_b200 import workloads as wl

pytestmark = pytest.mark.gpu

# (N,C,H,W,K,R,S,stride,pad,relu): points 127 / 128 / 129 per call, channels around 32 and 64, windows on both sides of the
# largest that is staged through shared memory (36 taps; beyond and at multiples of 8, runs of 8 taps with and without a remainder), filter counts that leave a last block nearly empty
SHAPES = [
    (1, 31, 1, 127, 17, 1, 1, 1, 0, 0),
    (1, 33, 8, 16, 9, 1, 1, 1, 0, 1),
    (3, 64, 1, 43, 65, 1, 1, 1, 0, 1),
    (1, 770, 3, 5, 100, 1, 1, 1, 0, 0),
    (2, 65, 9, 9, 33, 3, 3, 1, 1, 1),
    (1, 40, 12, 13, 24, 6, 6, 1, 2, 1),
    (1, 20, 14, 15, 16, 7, 7, 2, 3, 1),
    (1, 35, 11, 11, 8, 11, 11, 1, 5, 0),
    (2, 33, 10, 12, 9, 4, 10, 1, 2, 0),
    (1, 40, 9, 12, 19, 9, 11, 1, 4, 1),
    (2, 33, 10, 12, 9, 4, 4, 1, 1, 0),           # 16 and 32 taps: runs too
    (1, 70, 9, 12, 19, 8, 4, 1, 2, 1),
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("math", [0, 3, 4])          # TF32, error-compensated TF32, fp16 storage
@pytest.mark.parametrize("bind", [False, True])
def test_staged_operands_exact(shape, math, bind):
    N, C, H, W, K, R, S, *_ = shape
    x, w, b = wl.integers(9400, (N, C, H, W)), wl.integers(9401, (K, C, R, S)), wl.integers(9402, (K,))
    got, desc = run_planned(shape, x, w, b, variant=1 if R * S == 1 else 2, math=math, tile_id=0, s2d=0, bind=bind)
    assert "igemm_128x64" in desc
    np.testing.assert_array_equal(got.astype(np.float64), oracle_out(shape, x, w, b), err_msg=desc)
