"""Which filters a plan computes with: those the call hands over, whatever the plan was tuned with or saw before; and what
FP32 plans hold.  Integer-valued operands make every sum exact."""
import ctypes

import numpy as np
import pytest

from helpers import oracle_out
from paper_1606_00094_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _ints(shape, seed):
    N, C, H, W, K, R, S, *_ = shape
    return wl.integers(seed, (N, C, H, W)), wl.integers(seed + 1, (K, C, R, S)), wl.integers(seed + 2, (K,))


def test_tuned_fp32_plan_does_not_keep_the_tuners_filters():
    """The tuner's scratch buffers are freed when it is done; blocks of the same size that a program allocates next get their
    addresses, and filters that it puts there are not the tuner's.  (Every call brings other filters than the one before it.)"""
    import torch
    from paper_1606_00094_b200 import binding as B
    shape = (20, 256, 13, 13, 384, 3, 3, 1, 1, 1)
    x, w, b = _ints(shape, 9700)
    dx, db = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    sides = [(torch.from_numpy(f).cuda(), torch.from_numpy(oracle_out(shape, x, f, b).astype(np.float32)).cuda()) for f in (w, wl.integers(9703, w.shape))]
    out = torch.empty_like(sides[0][1])
    torch.cuda.synchronize()
    cudart = ctypes.CDLL("libcudart.so.12")
    o = B.boda_plan_opts_default()
    o.math, o.tune = B.BODA_MATH_FP32, 1
    handle = B.boda_conv_plan_create(shape, o)
    assert "direct_nhwc" in B.boda_conv_plan_describe(handle)
    blocks = []
    try:
        for _ in range(32):
            p = ctypes.c_void_p()
            assert cudart.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(w.nbytes)) == 0
            blocks.append(p)
        ws = torch.empty(B.boda_conv_plan_workspace_bytes(handle), dtype=torch.uint8, device="cuda")
        for i, p in enumerate(blocks):
            filt, want = sides[i & 1]
            assert cudart.cudaMemcpy(p, ctypes.c_void_p(filt.data_ptr()), ctypes.c_size_t(w.nbytes), ctypes.c_int(3)) == 0      # device to device
            B.boda_conv_fwd_planned(handle, dx, p.value, db, out, ws)
            assert torch.equal(out, want)
    finally:
        torch.cuda.synchronize()
        B.boda_conv_plan_destroy(handle)
        for p in blocks:
            cudart.cudaFree(p)


# what the rule picks with workspace: split operands on the tensor cores, and FP32 arithmetic over a staged input
BY_RULE = [((20, 256, 13, 13, 384, 3, 3, 1, 1, 1), "direct_nhwc_x3_128x"), ((3, 328, 11, 13, 9, 11, 11, 4, 0, 1), "direct_nhwc_128x")]


@pytest.mark.parametrize("shape,tile", [(BY_RULE[0][0], -1), (BY_RULE[1][0], -1), ((3, 36, 13, 13, 97, 3, 3, 1, 1, 1), 20), ((3, 36, 13, 13, 97, 3, 3, 1, 1, 1), 2)])
def test_fp32_plans_read_their_filters_on_every_call(shape, tile):
    """Binding an FP32 plan keeps nothing: filters written anew in place, and other filters in between, are what the next call uses."""
    import torch
    from paper_1606_00094_b200 import binding as B
    x, w, b = _ints(shape, 9710)
    w2 = wl.integers(9713, w.shape)
    dx, db = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    bound, other = torch.from_numpy(w).cuda(), torch.from_numpy(w2).cuda()
    ref, ref2 = oracle_out(shape, x, w, b), oracle_out(shape, x, w2, b)
    plan = B.ConvPlan(shape, math=B.BODA_MATH_FP32, variant=B.BODA_VARIANT_DIRECT, tile_id=tile)
    assert tile >= 0 or dict(BY_RULE)[shape] in plan.describe()
    plan.bind_filters(bound)
    for filt, want in ((bound, ref), (other, ref2), (bound, ref)):
        np.testing.assert_array_equal(plan(dx, filt, db).cpu().numpy().astype(np.float64), want, err_msg=plan.describe())
    bound.copy_(other)
    np.testing.assert_array_equal(plan(dx, bound, db).cpu().numpy().astype(np.float64), ref2, err_msg=plan.describe())
    plan.close()


@pytest.mark.parametrize("shape,variant,tile,math", [
    ((3, 64, 13, 13, 97, 3, 3, 1, 1, 1), 2, 2, 0),           # im2col
    ((3, 64, 13, 13, 97, 3, 3, 1, 1, 1), 2, 2, 3),
    ((3, 64, 13, 13, 97, 3, 3, 1, 1, 1), 2, 31, 3),          # split operands
    ((3, 64, 13, 13, 97, 3, 3, 1, 1, 1), 2, 34, 3),
    ((3, 64, 13, 13, 97, 3, 3, 1, 1, 1), 2, 6, 0),           # halo
    ((3, 64, 13, 13, 97, 3, 3, 1, 1, 1), 2, 17, 0),          # gather
    ((2, 3, 67, 67, 80, 11, 11, 4, 0, 1), 2, 24, 0),         # first layer
    ((3, 64, 12, 12, 97, 1, 1, 1, 0, 1), 1, 20, 0),          # 1x1 from NCHW
    ((3, 64, 13, 13, 97, 3, 3, 1, 1, 1), 2, 28, 4),          # CTA pairs, fp16
])
def test_other_filters_between_calls_with_the_bound_ones(shape, variant, tile, math):
    """A tensor-core plan has room for one packed copy: a call with other filters writes over it, so the bound ones are packed again."""
    import torch
    from paper_1606_00094_b200 import binding as B
    x, w, b = _ints(shape, 9720)
    w2 = wl.integers(9723, w.shape)
    dx, db = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    bound, other = torch.from_numpy(w).cuda(), torch.from_numpy(w2).cuda()
    ref, ref2 = oracle_out(shape, x, w, b), oracle_out(shape, x, w2, b)
    plan = B.ConvPlan(shape, math=math, variant=variant, tile_id=tile)
    plan.bind_filters(bound)
    for filt, want in ((bound, ref), (other, ref2), (bound, ref), (other, ref2)):
        np.testing.assert_array_equal(plan(dx, filt, db).cpu().numpy().astype(np.float64), want, err_msg=plan.describe())
    plan.bind_filters(bound)
    np.testing.assert_array_equal(plan(dx, bound, db).cpu().numpy().astype(np.float64), ref, err_msg=plan.describe())
    plan.close()


# few filters, or little work: layers that the one-call entry point runs on the FP32 kernel
ONE_CALL_FP32 = [(1, 370, 23, 23, 10, 9, 9, 1, 4, 1), (88, 651, 14, 14, 3, 7, 7, 2, 0, 1)]


@pytest.mark.parametrize("shape", ONE_CALL_FP32)
def test_one_call_fp32_layers_hold_no_buffers(shape):
    """Calls of one shape share a cached plan: a kernel that stages its operands there would let two streams overwrite each other's,
    so these layers run on the one kernel that reads them where they lie."""
    import torch
    from paper_1606_00094_b200 import binding as B
    x, w, b = _ints(shape, 9730)
    dx, dw, db = (torch.from_numpy(t).cuda() for t in (x, w, b))
    args = dict(stride=shape[7], pad=shape[8], relu=True)
    B.conv_fwd(dx, dw, db, **args)
    before = B.boda_kernel_launch_count()
    got = B.conv_fwd(dx, dw, db, **args)
    assert B.boda_kernel_launch_count() - before == 1
    np.testing.assert_array_equal(got.cpu().numpy().astype(np.float64), oracle_out(shape, x, w, b))


def test_one_call_fp32_layers_on_two_streams():
    import torch
    from paper_1606_00094_b200 import binding as B
    shape = ONE_CALL_FP32[0]
    sides = []
    for seed in (9731, 9741):
        x, w, b = _ints(shape, seed)
        sides.append((torch.cuda.Stream(), [torch.from_numpy(t).cuda() for t in (x, w, b)],
                      torch.from_numpy(oracle_out(shape, x, w, b).astype(np.float32)).cuda(), []))
    torch.cuda.synchronize()
    for _ in range(50):
        for stream, (dx, dw, db), _, outs in sides:
            with torch.cuda.stream(stream):
                outs.append(B.conv_fwd(dx, dw, db, stride=shape[7], pad=shape[8], relu=True))
    torch.cuda.synchronize()
    for _, _, want, outs in sides:
        assert all(torch.equal(o, want) for o in outs)


@pytest.mark.parametrize("shape,name", BY_RULE)
def test_fp32_plan_runs_without_workspace(shape, name):
    """FP32 plans picked by rule take workspace where they can use it and run without (or with one off its alignment) on the
    kernel that needs none; only a forced staged tile insists."""
    import torch
    from paper_1606_00094_b200 import binding as B
    x, w, b = _ints(shape, 9740)
    dx, dw, db = (torch.from_numpy(t).cuda() for t in (x, w, b))
    want = oracle_out(shape, x, w, b)
    out = torch.empty(want.shape, device="cuda")
    plan = B.ConvPlan(shape, math=B.BODA_MATH_FP32)
    assert name in plan.describe()
    for ws in (None, plan.workspace, plan.workspace[4:], None):
        out.fill_(float("nan"))
        B.boda_conv_fwd_planned(plan.handle, dx, dw, db, out, ws)
        np.testing.assert_array_equal(out.cpu().numpy().astype(np.float64), want)
    plan.close()
    refused = []

    def no_memory(*size, **kw):
        refused.append(size)
        raise torch.OutOfMemoryError("no memory")
    with pytest.MonkeyPatch.context() as patch:
        patch.setattr(torch, "empty", no_memory)
        plan = B.ConvPlan(shape, math=B.BODA_MATH_FP32)
        with pytest.raises(torch.OutOfMemoryError):                          # a forced tile: no other kernel to fall back to
            B.ConvPlan(shape, math=1, variant=0, tile_id=24)
        if shape[4] >= 16:
            with pytest.raises(torch.OutOfMemoryError):
                B.ConvPlan(shape, math=3)
    assert len(refused) >= 2 and plan.workspace is None
    np.testing.assert_array_equal(plan(dx, dw, db).cpu().numpy().astype(np.float64), want)
    plan.close()
    forced = B.ConvPlan(shape, math=B.BODA_MATH_FP32, variant=B.BODA_VARIANT_DIRECT, tile_id=18)
    with pytest.raises(B.BodaError) as e:
        B.boda_conv_fwd_planned(forced.handle, dx, dw, db, out, None)
    assert e.value.status == B.BODA_ERR_NOMEM
    forced.close()
