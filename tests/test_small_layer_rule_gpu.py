"""Small layers that the automatic rule leaves to the FP32 kernel in place, and neighbours that it does not: what the plan is, that nothing else
about the call changes, and that forced variants, modes and chains keep their kernels."""
import numpy as np
import pytest

from helpers import FP32_TOL, TF32_TOL, assert_parity, oracle_out, run_planned
from paper_1606_00094_b200 import workloads as wl

pytestmark = pytest.mark.gpu

# (N,C,H,W,K,R,S,stride,pad,relu), measured times in place / tensor cores (us)
IN_PLACE = [
    (2, 355, 7, 7, 25, 1, 1, 1, 0, 1),           # 4.0 / 7.8
    (2, 505, 15, 15, 31, 1, 1, 1, 0, 0),         # 4.8 / 9.1
    (4, 9, 15, 15, 29, 5, 5, 1, 2, 1),           # 5.0 / 10.6
    (1, 17, 19, 21, 105, 3, 3, 2, 1, 1),         # 4.4 / 7.9
    (1, 7, 39, 42, 16, 1, 1, 1, 0, 1),           # 3.1 / 5.8
    (38, 10, 35, 35, 28, 1, 1, 1, 0, 1),         # 5.7 / 11.4: one chunk, many points
    (40, 16, 41, 43, 29, 1, 1, 1, 0, 1),         # 7.3 / 13.9
]
TENSOR = [
    (5, 480, 14, 14, 192, 1, 1, 1, 0, 1),        # 11.5 / 6.5
    (5, 174, 28, 28, 28, 1, 1, 1, 0, 1),         # 7.3 / 5.1
    (20, 256, 13, 13, 384, 3, 3, 1, 1, 1),
    (1, 3, 227, 227, 96, 11, 11, 4, 0, 1),       # more taps than the bounds mask holds
]


def _tensors(shape):
    N, C, H, W, K, R, S, *_ = shape
    return wl.half_normal(1, (N, C, H, W)), wl.normal(2, (K, C, R, S), 0, (2.0 / (C * R * S)) ** 0.5), wl.normal(3, (K,), 0, 0.01)


@pytest.mark.parametrize("shape", IN_PLACE)
def test_small_layers_run_in_place(shape):
    import torch
    from paper_1606_00094_b200 import binding as B
    x, w, b = _tensors(shape)
    ref = oracle_out(shape, x, w, b)
    for bind in (False, True):
        got, desc = run_planned(shape, x, w, b, bind=bind)
        assert "variant=direct" in desc and "workspace=0" in desc
        assert_parity(got, ref, FP32_TOL, desc)
    args = [torch.from_numpy(t).cuda() for t in (x, w, b)]
    call = lambda: B.conv_fwd(*args, stride=shape[7], pad=shape[8], relu=bool(shape[9]))
    call()
    before = B.boda_kernel_launch_count()
    got = call()
    assert B.boda_kernel_launch_count() - before == 1
    assert_parity(got.cpu().numpy(), ref, FP32_TOL)
    variant = 1 if shape[5] * shape[6] == 1 else 2
    for kw in (dict(variant=variant), dict(variant=variant, math=2)):
        got, desc = run_planned(shape, x, w, b, **kw)
        assert "math=tf32" in desc
        assert_parity(got, ref, TF32_TOL, desc)


# layers that the run-time compiled tiles suit
SUIT_COMPILED = [(1, 7, 39, 42, 16, 1, 1, 1, 0, 1), (2, 8, 25, 25, 24, 1, 1, 1, 0, 1), (3, 30, 13, 13, 100, 1, 1, 1, 0, 1), (2, 20, 40, 40, 16, 3, 3, 1, 1, 1)]


@pytest.mark.parametrize("shape", SUIT_COMPILED)
def test_the_rule_compiles_nothing_at_run_time(shape):
    """A compilation would sit in the first one-call of a shape, or in a plan whose tensor-core kernel needed none."""
    from paper_1606_00094_b200 import binding as B
    plan = B.ConvPlan(shape)
    desc = plan.describe()
    plan.close()
    assert "rtc" not in desc
    x, w, b = _tensors(shape)
    got, desc = run_planned(shape, x, w, b)
    assert_parity(got, oracle_out(shape, x, w, b), FP32_TOL if "variant=direct" in desc else TF32_TOL, desc)


@pytest.mark.parametrize("shape", TENSOR)
def test_layers_that_stay_on_the_tensor_cores(shape):
    from paper_1606_00094_b200 import binding as B
    assert "math=tf32" in B.ConvPlan(shape).describe()


def test_chains_keep_their_kernels():
    from paper_1606_00094_b200 import binding as B
    from paper_1606_00094_b200.stack import ConvStack
    ops = [wl.StackOp("conv", wl.ConvShape(2, 40, 13, 13, 64, 3, 3, 1, 1)), wl.StackOp("conv", wl.ConvShape(2, 64, 13, 13, 48, 1, 1, 1, 0))]
    assert "variant=direct" in B.ConvPlan((2, 64, 13, 13, 48, 1, 1, 1, 0, 1)).describe()
    params = [(wl.integers(1 + i, (o.shape.K, o.shape.C, o.shape.R, o.shape.S)), wl.integers(5 + i, (o.shape.K,))) for i, o in enumerate(ops)]
    stack = ConvStack(ops, params)
    assert all("math=tf32" in d for d in stack.describe())
    stack.close()


def test_matrix_products_of_small_extents():
    import torch
    from paper_1606_00094_b200 import binding as B
    for M, N, K in ((93, 157, 221), (64, 64, 64), (313, 324, 84)):        # 9.5 -> 4.0 us for the first
        A, Bm, C = torch.randn(M, K, device="cuda"), torch.randn(K, N, device="cuda"), torch.empty(M, N, device="cuda")
        B.boda_sgemm(A, Bm, C, M, N, K)
        before = B.boda_kernel_launch_count()
        B.boda_sgemm(A, Bm, C, M, N, K)
        assert B.boda_kernel_launch_count() - before == 1
        ref = A.double() @ Bm.double()
        assert ((C.double() - ref).norm() / ref.norm()).item() <= FP32_TOL
