"""The calls that a user of this library makes, as cases that can be timed and compared.

A convolution layer is trained by three passes per step (fprop, bprop, accGrad) on a plan
that the program keeps, so most cases are such a step: from a layer whose whole step is
launch latency to planes of 128 x 128.  The others are the remaining ways to call the
library: inference without a workspace, the exact FP32 contraction, spectrum reuse,
spatial tiling and the bare batched transforms in both directions.

Layer shapes are the benchmark configs and the paper's Table 2 layers, `draw` covers the
parameter sweep's ranges with the sizes in between.
"""
from __future__ import annotations

import math

import torch

import paper_1412_7580_b200 as fc
from paper_1412_7580_b200 import binding
from paper_1412_7580_b200 import workloads as wl


def _layer(name, S, f, fp, h, w, kh, kw, **options):
    """A training step of one layer; `options` are those of `_layer_plan`."""
    case = dict(kind="step", S=S, f=f, fp=fp, h=h, w=w, kh=kh, kw=kw, n=max(8, wl.next_pow2(max(h, w))),
                math="auto", reuse=False, tile=0, accumulate=False)
    case.update(options)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # Smallest layer in use: a few planes, every kernel is launch latency and host path.
        _layer("tiny_step", 8, 4, 8, 16, 16, 3, 3),
        # Inference of one image inside a program that cannot allocate (fprop alone, built-in scratch).
        _layer("infer_noalloc", 1, 16, 64, 57, 57, 5, 5, kind="infer"),
        # Odd counts, rectangular planes and kernels; a training loop that keeps the spectra
        # between the passes of a step and adds to its weight gradient.
        _layer("ragged_reuse_step", 50, 67, 90, 27, 29, 5, 3, reuse=True, accumulate=True),
        # The middle layers of an AlexNet-like network: many planes of 31 x 31.
        _layer("mid_step", 128, 96, 256, 31, 31, 5, 5),
        # Large kernels on 64 x 64 planes: where the FFT method beats direct convolution most.
        _layer("large_kernel_step", 128, 64, 64, 64, 64, 11, 11),
        # Deep layers: small planes, many features, dominated by the contraction.
        _layer("deep_step", 128, 384, 384, 13, 13, 3, 3),
        # The same kind of step where TF32 is not accurate enough: exact FP32 contraction.
        _layer("mid_fp32_step", 128, 96, 256, 31, 31, 5, 5, math="fp32"),
        # Early layers with full-size planes (n = 128).
        _layer("wide_planes_step", 64, 64, 64, 128, 128, 5, 5),
        # First layer of a network: three input planes, 128 x 128 images, 11 x 11 kernels.
        _layer("first_layer_step", 128, 3, 96, 128, 128, 11, 11),
        # Large planes with small kernels and many features: the plan chooses a tile basis.
        _layer("tiled_step", 16, 256, 256, 128, 128, 3, 3, tile=binding.TILE_AUTO),
        # The transforms alone, forward with zero-padding and inverse with crop, two-dimensional ...
        dict(name="fft2d_round_trip", kind="fft2d", batch=8191, h=57, w=57, n=64),
        # ... and one-dimensional.
        dict(name="fft1d_round_trip", kind="fft1d", batch=262143, len=250, n=256),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _cost(case):
    """What a case moves, spectra included: keeps drawn cases within the largest listed one."""
    if case["kind"] == "fft1d":
        return case["batch"] * (8.0 * case["len"] + 16.0 * (case["n"] // 2 + 1))
    if case["kind"] == "fft2d":
        return case["batch"] * (8.0 * case["h"] * case["w"] + 16.0 * case["n"] * (case["n"] // 2 + 1))
    S, f, fp, n = case["S"], case["f"], case["fp"], case["n"]
    bins = n * (n // 2 + 1)
    spectra = 4 * 8.0 * bins * (S * f + f * fp + S * fp)
    # an FP32 contraction is bound by its arithmetic: bytes that take as long
    flops = 24.0 * bins * S * f * fp
    return spectra + (flops / 8.0 if case["math"] == "fp32" else flops / 60.0)


def draw(rng):
    # the first layer takes longest of the listed cases (its transforms are those of n = 128)
    limit = next(_cost(c) for c in listed() if c["name"] == "first_layer_step")
    while True:
        kind = rng.choices(["step", "infer", "fft2d", "fft1d"], weights=[16, 2, 3, 3])[0]
        if kind == "fft1d":
            n = rng.choice([8, 16, 32, 64, 128, 256])
            case = dict(kind=kind, batch=_log_int(rng, 64, 2000000), len=rng.randint(n // 2 + 1, n), n=n)
        elif kind == "fft2d":
            n = rng.choice([8, 16, 32, 64, 128])
            case = dict(kind=kind, batch=_log_int(rng, 16, 300000), h=rng.randint(n // 2 + 1, n),
                        w=rng.randint(n // 2 + 1, n), n=n)
        else:
            h = _log_int(rng, 13, 128)
            w = h if rng.random() < 0.6 else max(13, min(128, int(round(h * rng.uniform(0.7, 1.4)))))
            kh = rng.choice([k for k in wl.SWEEP_K if k <= h])
            kw = kh if rng.random() < 0.8 else rng.choice([k for k in wl.SWEEP_K if k <= w])
            case = _layer(None, _log_int(rng, 1, 128), _log_int(rng, 1, 384), _log_int(rng, 1, 384), h, w, kh, kw,
                          kind=kind)
            if kind == "infer":
                case.update(S=_log_int(rng, 1, 8), f=_log_int(rng, 1, 64), fp=_log_int(rng, 1, 64))
                if fc.conv_plan_workspace_bytes(_layer_plan(case)) > binding.NOALLOC_BYTES:
                    continue
            else:
                option = rng.choices(["none", "fp32", "reuse", "tile", "accumulate"], weights=[10, 2, 2, 3, 2])[0]
                case.update(math="fp32" if option == "fp32" else "auto", reuse=option == "reuse",
                            tile=binding.TILE_AUTO if option == "tile" else 0, accumulate=option == "accumulate")
        if _cost(case) <= limit:
            return case


def _layer_plan(case):
    plan = fc.conv_plan(case["S"], case["f"], case["fp"], case["h"], case["w"], case["kh"], case["kw"], case["n"])
    if case["math"] == "fp32":
        fc.conv_plan_set_math(plan, binding.MATH_FP32)
    if case["reuse"]:
        fc.conv_plan_set_spectrum_reuse(plan, True)
    if case["tile"]:
        fc.conv_plan_set_tiling(plan, case["tile"])
    return plan


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))

    def uniform(*dims):
        return torch.rand(dims, generator=gen, device="cuda").mul_(2.0).sub_(1.0)

    def normal(std, *dims):
        return torch.randn(dims, generator=gen, device="cuda").mul_(std)

    def empty(*dims):
        return torch.empty(dims, device="cuda")

    state = dict(case=case)
    if case["kind"] == "fft1d":
        bins = case["n"] // 2 + 1
        state.update(x=uniform(case["batch"], case["len"]), spectrum=empty(case["batch"], bins, 2),
                     back=empty(case["batch"], case["len"]))
        return state
    if case["kind"] == "fft2d":
        n = case["n"]
        state.update(x=uniform(case["batch"], case["h"], case["w"]), spectrum=empty(case["batch"], n, n // 2 + 1, 2),
                     back=empty(case["batch"], case["h"], case["w"]))
        return state
    S, f, fp, h, w, kh, kw = (case[k] for k in ("S", "f", "fp", "h", "w", "kh", "kw"))
    oh, ow = h - kh + 1, w - kw + 1
    plan = _layer_plan(case)
    # activations uniform, weights scaled by the fan-in, output gradients normal
    state.update(plan=plan, x=uniform(S, f, h, w), w=normal((f * kh * kw) ** -0.5, fp, f, kh, kw),
                 y=empty(S, fp, oh, ow))
    if case["kind"] == "infer":
        return state
    fc.conv_plan_alloc_workspace(plan)
    state.update(dy=normal(1.0, S, fp, oh, ow), dx=empty(S, f, h, w),
                 # a gradient that is added to starts from an earlier microbatch's
                 dw=empty(fp, f, kh, kw))
    if case["accumulate"]:
        state["dw_before"] = normal((S * oh * ow) ** 0.5, fp, f, kh, kw)
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "fft1d":
        fc.fft1d_r2c(state["x"], state["spectrum"], case["n"])
        fc.fft1d_c2r(state["spectrum"], state["back"], case["n"], 1.0 / case["n"])
        return state["spectrum"], state["back"]
    if case["kind"] == "fft2d":
        fc.fft2d_r2c(state["x"], state["spectrum"], case["n"])
        fc.fft2d_c2r(state["spectrum"], state["back"], case["n"], 1.0 / case["n"] ** 2)
        return state["spectrum"], state["back"]
    plan = state["plan"]
    if case["kind"] == "infer":
        fc.conv_fprop_noalloc(plan, state["x"], state["w"], state["y"])
        return state["y"]
    fc.conv_fprop(plan, state["x"], state["w"], state["y"])
    fc.conv_bprop(plan, state["dy"], state["w"], state["dx"])
    if case["accumulate"]:
        state["dw"].copy_(state["dw_before"])
    fc.conv_accgrad(plan, state["dy"], state["x"], state["dw"], accumulate=case["accumulate"])
    return state["y"], state["dx"], state["dw"]


def work(case):
    """Tensors in and out once; the transforms' 2.5 N log2 N operations per plane and the
    contraction's eight per complex multiply-add (Table 1 of the paper), over the basis in use."""
    if case["kind"] == "fft1d":
        n, batch = case["n"], case["batch"]
        return dict(bytes=batch * (8.0 * case["len"] + 8.0 * (n // 2 + 1)), flops=2 * batch * 2.5 * n * math.log2(n))
    if case["kind"] == "fft2d":
        n, batch = case["n"], case["batch"]
        return dict(bytes=batch * (8.0 * case["h"] * case["w"] + 8.0 * n * (n // 2 + 1)),
                    flops=2 * batch * 2.5 * n * n * math.log2(n * n))
    S, f, fp, h, w, kh, kw = (case[k] for k in ("S", "f", "fp", "h", "w", "kh", "kw"))
    oh, ow = h - kh + 1, w - kw + 1
    x, wt, y = S * f * h * w, fp * f * kh * kw, S * fp * oh * ow
    if case["kind"] == "infer":
        passes, nbytes = 1, 4.0 * (x + wt + y)
    else:
        # x, w, dy in; y, dx, dw out (and the gradient that is added to)
        passes, nbytes = 3, 4.0 * (2 * x + 2 * wt + 2 * y + (wt if case["accumulate"] else 0))
    n, windows = case["n"], 1
    if case["tile"]:
        basis = fc.conv_plan_tile_basis(_layer_plan(case))
        if basis:
            n = basis
            windows = -(-oh // (n - kh + 1)) * -(-ow // (n - kw + 1))
    bins = n * (n // 2 + 1)
    planes = windows * S * (f + fp) + f * fp
    fft = 2.5 * n * n * math.log2(n * n) * planes
    return dict(bytes=nbytes, flops=passes * (fft + 8.0 * bins * windows * S * f * fp))


def tolerance(case):
    # four times the largest error seen against float64: 2e-7 (transforms), 7e-7 (FP32 passes),
    # 7.7e-4 (TF32 operands); a step's outputs are judged by its least exact pass
    if case["kind"] in ("fft1d", "fft2d"):
        return {"rel": 8e-7}
    passes = [0] if case["kind"] == "infer" else [0, 1, 2]
    plan = _layer_plan(case)
    if any(fc.conv_plan_pass_math(plan, p) == binding.MATH_TF32 for p in passes):
        return {"rel": 3e-3}
    return {"rel": 3e-6}
