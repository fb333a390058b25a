"""The work a user of this library has it do, as a list of timed cases: single layers through a plan, one-call layers, the
matrix product and whole chains, from one 32x32 image to a batch of 128 through five convolutions.

Sizes are those of the benchmark configurations (`workloads.CONFIGS`), of the layers of the AlexNet-shaped stack, of the
matrix-product table and of the tests, at the batch sizes 1, 5 and 20 of the paper, and above them where throughput is what
counts.  Inputs have the distributions of `workloads.py` (uniform images, half-normal activations, He-normal filters, small
biases), made on the GPU from the seed.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_1606_00094_b200 import binding as B
from paper_1606_00094_b200 import workloads as wl
from paper_1606_00094_b200.stack import ConvStack

MATH = {"auto": B.BODA_MATH_AUTO, "fp32": B.BODA_MATH_FP32, "tf32x3": B.BODA_MATH_TF32X3, "f16": B.BODA_MATH_F16}

#: Largest drawn layer (the largest listed case is the batch-128 chain: 275.6 GFLOP).
MOST_LAYER_FLOPS = {"auto": 60e9, "f16": 60e9, "tf32x3": 20e9, "fp32": 6e9}
MOST_LAYER_BYTES = 300e6


def layer(kind, N, C, H, W, K, R, S, stride, pad, math_mode="auto"):
    """kind: "plan" (explicit plan, filters bound once) or "onecall" (`conv_fwd`, everything handed over on every call)."""
    return {"kind": kind, "N": N, "C": C, "H": H, "W": W, "K": K, "R": R, "S": S, "stride": stride, "pad": pad, "math": math_mode}


def listed():
    return [
        # one small image through one small layer: what a call costs when the arithmetic is next to nothing
        {"name": "small3x3_b1", **layer("plan", 1, 3, 32, 32, 16, 3, 3, 1, 1)},
        # first layer of a network on one image (large window, stride 4, three channels): latency of a single request
        {"name": "first_11x11_b1", **layer("plan", 1, 3, 227, 227, 96, 11, 11, 4, 0)},
        # 1x1 layer of an inception block, small batch: ordinary request batching
        {"name": "inception_1x1_b5", **layer("plan", 5, 480, 14, 14, 192, 1, 1, 1, 0)},
        # the same layer at a throughput batch: the memory-bound end
        {"name": "inception_1x1_b256", **layer("plan", 256, 480, 14, 14, 192, 1, 1, 1, 0)},
        # 3x3 layer in the middle of a network, batch 20: the ordinary compute-bound layer
        {"name": "conv3_b20", **layer("plan", 20, 256, 13, 13, 384, 3, 3, 1, 1)},
        # ragged extents and channel counts through the one-call entry point: filters change hands on every call
        {"name": "odd_3x3_onecall", **layer("onecall", 7, 100, 29, 31, 130, 3, 3, 1, 1)},
        # 5x5 layer with 16-bit operand storage
        {"name": "conv2_b20_f16", **layer("plan", 20, 96, 27, 27, 256, 5, 5, 1, 2, "f16")},
        # 3x3 layer with error-compensated TF32, request batch
        {"name": "conv3_b5_tf32x3", **layer("plan", 5, 256, 13, 13, 384, 3, 3, 1, 1, "tf32x3")},
        # the ordinary layer for a caller who insists on FP32 arithmetic
        {"name": "conv3_b20_fp32", **layer("plan", 20, 256, 13, 13, 384, 3, 3, 1, 1, "fp32")},
        # matrix product between the table's sizes, rows of B not a multiple of 16 bytes
        {"name": "sgemm_ragged", "kind": "sgemm", "M": 1000, "N": 1301, "K": 770},
        # the AlexNet-shaped chain at the benchmark's batch, one graph launch
        {"name": "stack_b20", "kind": "stack", "N": 20},
        # and at a throughput batch: the largest work
        {"name": "stack_b128", "kind": "stack", "N": 128},
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], uniform over the logarithm."""
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        kind = rng.choice(["small", "first", "one", "one", "window", "window", "onecall", "modes", "modes", "sgemm", "stack"])
        if kind == "sgemm":
            return {"kind": "sgemm", "M": _log(rng, 64, 2048), "N": _log(rng, 64, 2048), "K": _log(rng, 64, 2048)}
        if kind == "stack":
            return {"kind": "stack", "N": _log(rng, 1, 127)}
        if kind == "small":
            ksz = rng.choice([1, 3, 5])
            hw = rng.randint(12, 64)
            c = layer("plan", _log(rng, 1, 8), rng.randint(1, 16), hw, hw + rng.randint(0, 3), rng.randint(4, 32), ksz, ksz, 1, ksz // 2)
        elif kind == "first":
            ksz, stride = rng.choice([(11, 4), (7, 2), (5, 2), (3, 1), (5, 1), (3, 2)])
            hw = rng.randint(64, 240)
            c = layer("plan", _log(rng, 1, 64), 3, hw, hw, rng.choice([32, 48, 64, 96]), ksz, ksz, stride, rng.choice([0, ksz // 2]))
        elif kind == "one":
            hw = rng.choice([6, 7, 13, 14, 15, 27, 28, 54, 56])
            c = layer("plan", _log(rng, 1, 256), _log(rng, 64, 1024), hw, hw, _log(rng, 16, 512), 1, 1, 1, 0)
        else:
            ksz, stride = rng.choice([(3, 1), (3, 1), (5, 1), (3, 2)])
            hw = rng.randint(6, 56)
            c = layer("onecall" if kind == "onecall" else "plan", _log(rng, 1, 64), _log(rng, 16, 512), hw, hw + rng.randint(0, 2),
                      _log(rng, 32, 512), ksz, ksz, stride, ksz // 2, rng.choice(["f16", "tf32x3", "fp32"]) if kind == "modes" else "auto")
        w = work(c)
        if w["flops"] <= MOST_LAYER_FLOPS[c["math"]] and w["bytes"] <= MOST_LAYER_BYTES:
            return c


def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32)


def _he(gen, K, C, R, S):
    return _randn(gen, K, C, R, S) * math.sqrt(2.0 / (C * R * S))


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["kind"] == "sgemm":
        M, N, K = case["M"], case["N"], case["K"]
        return SimpleNamespace(kind="sgemm", M=M, N=N, K=K, a=_randn(gen, M, K), b=_randn(gen, K, N),
                               c=torch.empty(M, N, device="cuda"))
    if case["kind"] == "stack":
        ops = wl.alexnet_stack(case["N"])
        params = []
        for op in ops:
            if op.kind == "conv":
                s = op.shape
                params.append((_he(gen, s.K, s.C, s.R, s.S).cpu().numpy(), (_randn(gen, s.K) * 0.01).cpu().numpy()))
        x = torch.rand(case["N"], 3, 227, 227, generator=gen, device="cuda")
        return SimpleNamespace(kind="stack", stack=ConvStack(ops, params), x=x)
    N, C, H, W, K, R, S = (case[k] for k in "NCHWKRS")
    # images are uniform, what comes out of an earlier layer is half-normal
    x = torch.rand(N, C, H, W, generator=gen, device="cuda") if C == 3 else _randn(gen, N, C, H, W).abs()
    w, b = _he(gen, K, C, R, S), _randn(gen, K) * 0.01
    st = SimpleNamespace(kind=case["kind"], x=x, w=w, b=b, stride=case["stride"], pad=case["pad"])
    if case["kind"] == "plan":
        st.plan = B.ConvPlan((N, C, H, W, K, R, S, case["stride"], case["pad"], 1), math=MATH[case["math"]])
        st.plan.bind_filters(w)
    return st


def run(state):
    if state.kind == "plan":
        return state.plan(state.x, state.w, state.b)
    if state.kind == "onecall":
        return B.conv_fwd(state.x, state.w, state.b, stride=state.stride, pad=state.pad)
    if state.kind == "sgemm":
        B.boda_sgemm(state.a, state.b, state.c, state.M, state.N, state.K)
        return state.c
    return state.stack.forward(state.x)


def work(case):
    if case["kind"] == "sgemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 4 * (M * K + K * N + M * N), "flops": 2 * M * N * K}
    if case["kind"] == "stack":
        N, ops = case["N"], wl.alexnet_stack(case["N"])
        weights = sum(op.shape.K * (op.shape.C * op.shape.R * op.shape.S + 1) for op in ops if op.kind == "conv")
        return {"bytes": 4 * (N * 3 * 227 * 227 + weights + N * 256 * 6 * 6), "flops": wl.stack_flops(N)}
    s = wl.ConvShape(*(case[k] for k in ("N", "C", "H", "W", "K", "R", "S", "stride", "pad")))
    return {"bytes": s.min_bytes, "flops": s.flops}


def tolerance(case):
    # About four times the distance from the same path in 64 bits, over the listed cases and thirty drawn ones: TF32 layers
    # 2.5e-4 .. 5.6e-4 and the chain 5.7e-4 (largest single value 3.2e-3), fp16 storage 2.9e-4 (2.2e-3), error-compensated
    # TF32 0.5e-6 .. 4.2e-6 (1e-5), FP32 8e-7 (8e-6).
    mode = case.get("math", "auto")
    if mode == "fp32":
        return {"rel": 4e-6, "max": 4e-5}
    if mode == "tf32x3":
        return {"rel": 2e-5, "max": 8e-5}
    if mode == "f16":
        return {"rel": 1.2e-3, "max": 1e-2}
    return {"rel": 2e-3, "max": 1.3e-2}
