"""The calls whose speed this library is judged by: which shapes, which entry points, what counts as
the same result.

``listed()`` names twelve calls from one small plane to a 2^25-element one; ``draw(rng)`` makes more
of the same kinds and ranges.  A case is a dict:

    op      "mix"          whtmix.forward (whtmix.forward_padded where n < N)
            "sep"          whtmix.forward_separable (log gains; pads inside the library)
            "mix_train"    forward and backward of "mix", full gains
            "sep_train"    forward and backward of "sep"
            "block"        whtmix.block_forward
            "block_train"  whtmix.block_forward and whtmix.block_backward
    B, n, N, C   planes, stored tokens a plane, padded tokens (a power of two), channels
    dtype        "f32" or "bf16": X, Y, dY, dX (gains and their gradients are float32)
    autograd     mix_train only: through WHTMixFunction and torch.autograd.grad

Inference calls write into a buffer the program keeps; training calls get new outputs each time, as
autograd does.  The int32 mode is a checking mode of the library (exact, unnormalised), and no program
is expected to be waiting for it; it is left out.
"""
from __future__ import annotations

import math

import torch

from paper_2607_25234_gb300 import whtmix

TORCH_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}


def _case(name, op, B, n, N, C, dtype, autograd=False):
    return {"name": name, "op": op, "B": B, "n": n, "N": N, "C": C, "dtype": dtype, "autograd": autograd}


def listed():
    return [
        # the smallest mixer call a program makes: one map of 256 tokens; launch and latency
        _case("tiny_f32", "mix", 1, 256, 256, 64, "f32"),
        # batch-1 inference at a moderate token count (the middle of an isolated-mixer latency sweep)
        _case("single_bf16", "mix", 1, 4096, 4096, 64, "bf16"),
        # left + right rows of an epipolar stereo pair: many small planes
        _case("epipolar_bf16", "mix", 128, 512, 512, 128, "bf16"),
        # a batch of long sequences
        _case("longseq_f32", "mix", 32, 4096, 4096, 64, "f32"),
        # two quarter-resolution feature maps mixed globally, padded to 65536 tokens by the program
        _case("fullimage_bf16", "mix", 1, 65536, 65536, 128, "bf16"),
        # the paper's own form: log gains, 2 x 135 x 240 tokens padded inside the library
        _case("fullimage_log_gains_bf16", "sep", 1, 64800, 65536, 128, "bf16"),
        # the same maps at twice the resolution: 2 x 270 x 480 tokens padded to 262144
        _case("hires_bf16", "mix", 1, 259200, 262144, 128, "bf16"),
        # 8 x 8 token windows, forward and backward: planes far below one SM's memory
        _case("windows_train_f32", "mix_train", 200, 64, 64, 64, "f32"),
        # log gains trained on a batch of 4000-token sequences (ragged, padded inside the library)
        _case("longseq_log_gains_train_f32", "sep_train", 32, 4000, 4096, 64, "f32"),
        # a training step of the mixer with full gains, through autograd
        _case("train_bf16", "mix_train", 16, 8192, 8192, 256, "bf16", autograd=True),
        # the whole block (projections around the mixer) on the full image
        _case("block_fullimage_bf16", "block", 1, 65536, 65536, 128, "bf16"),
        # a training step of the whole block on a batch of medium maps
        _case("block_train_bf16", "block_train", 8, 4096, 4096, 128, "bf16"),
    ]


# log2 of the plane sizes each kind of call is made with, and of the most elements of a whole call
PLANE_BITS = {"mix": (10, 25), "sep": (12, 23), "mix_train": (10, 23), "sep_train": (12, 22),
              "block": (14, 23), "block_train": (14, 22)}
CALL_BITS = {"mix": 24.5, "sep": 24, "mix_train": 23.5, "sep_train": 23, "block": 24, "block_train": 22.5}


def draw(rng):
    op = rng.choice(sorted(PLANE_BITS))
    dtype = "bf16" if op.startswith("block") else rng.choice(["f32", "bf16"])
    C = rng.choice([64, 128, 256] if op.startswith("block") else [32, 64, 128, 256])
    lo, hi = PLANE_BITS[op]
    m = rng.randint(lo, hi)
    N = max(4, (1 << m) // C)
    m = (N * C).bit_length() - 1
    # half of the calls have a token count that is not a power of two (the block takes whole planes)
    n = N if op.startswith("block") or rng.random() < 0.5 else rng.randint(N // 2 + 1, N)
    B = max(1, int(2.0 ** rng.uniform(0.0, max(0.0, min(CALL_BITS[op] - m, 9.0)))))
    return {"op": op, "B": B, "n": n, "N": N, "C": C, "dtype": dtype,
            "autograd": op == "mix_train" and n == N and rng.random() < 0.5}


def _inputs(case, seed):
    """Activations and upstream gradients N(0, 1), gains around 1, log gains around 0 (the spread a
    trained mixer shows), projections of unit gain; the same values for the same seed."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    B, n, N, C = case["B"], case["n"], case["N"], case["C"]
    dt = TORCH_DTYPE[case["dtype"]]

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device=dev)

    t = {"x": normal(B, n, C).to(dt)}
    if case["op"].startswith("sep"):
        t["g_t"], t["g_c"] = 0.05 * normal(N), 0.05 * normal(C)
    else:
        t["g"] = 1.0 + 0.1 * normal(N, C)
    if case["op"].startswith("block"):
        t["w_in"] = (normal(C, C) / math.sqrt(C)).to(dt)
        t["w_out"] = (normal(C, C) / math.sqrt(C)).to(dt)
    if case["op"].endswith("train"):
        t["dy"] = normal(B, n, C).to(dt)
    return t


def prepare(case, seed):
    state = _inputs(case, seed)
    state["case"] = case
    if case["autograd"]:
        state["x"].requires_grad_(True)
        state["g"].requires_grad_(True)
    if not case["op"].endswith("train"):
        state["out"] = torch.empty_like(state["x"])
    return state


def run(state):
    s, case = state, state["case"]
    op, padded = case["op"], case["n"] < case["N"]
    if op == "mix":
        call = whtmix.forward_padded if padded else whtmix.forward
        return call(s["x"], s["g"], out=s["out"])
    if op == "sep":
        return whtmix.forward_separable(s["x"], s["g_t"], s["g_c"], out=s["out"])
    if op == "block":
        return whtmix.block_forward(s["x"], s["w_in"], s["g"], s["w_out"], out=s["out"])
    if op == "mix_train":
        if case["autograd"]:
            y = whtmix.WHTMixFunction.apply(s["x"], s["g"])
            dx, dg = torch.autograd.grad(y, (s["x"], s["g"]), s["dy"])
            return {"y": y.detach(), "dx": dx, "dg": dg}
        if padded:
            y = whtmix.forward_padded(s["x"], s["g"])
            dx, dg = whtmix.backward_padded(s["x"], s["g"], s["dy"])
        else:
            y = whtmix.forward(s["x"], s["g"])
            dx, dg = whtmix.backward(s["x"], s["g"], s["dy"])
        return {"y": y, "dx": dx, "dg": dg}
    if op == "sep_train":
        y = whtmix.forward_separable(s["x"], s["g_t"], s["g_c"])
        dx, dg_t, dg_c = whtmix.backward_separable(s["x"], s["g_t"], s["g_c"], s["dy"])
        return {"y": y, "dx": dx, "dg_t": dg_t, "dg_c": dg_c}
    y = whtmix.block_forward(s["x"], s["w_in"], s["g"], s["w_out"])
    dx, dw_in, dg, dw_out = whtmix.block_backward(s["x"], s["w_in"], s["g"], s["w_out"], s["dy"])
    return {"y": y, "dx": dx, "dw_in": dw_in, "dg": dg, "dw_out": dw_out}


def work(case):
    """Bytes: every input once, every output once.  Operations: 2 log2(N C) additions and one product
    for each element of a mixer map (its backward: one transform of X, two of dY, the gain and the
    products), 2 C for each element of a projection."""
    op, B, C = case["op"], case["B"], case["C"]
    es = 4 if case["dtype"] == "f32" else 2
    stored, plane = B * case["n"] * C, case["N"] * C
    L = B * plane
    bits = math.log2(plane)
    gains = 4 * (case["N"] + C) if op.startswith("sep") else 4 * plane
    nbytes, flops = 2 * stored * es + gains, L * (2 * bits + 1)
    if op.endswith("train"):
        nbytes += 2 * stored * es + gains          # dY, dX and the gains' gradients
        flops += L * (3 * bits + 3)
    if op.startswith("block"):
        nbytes += 2 * C * C * es
        flops += 2 * L * 2 * C
        if op == "block_train":
            nbytes += 2 * C * C * 4
            flops += 4 * L * 2 * C
    return {"bytes": int(nbytes), "flops": int(flops)}


def tolerance(case):
    """Relative 2-norm, about four times the distance from the 64-bit result that was measured:
    float32 butterflies over up to 25 bits; one rounding to bf16 at the store; in the block, roundings
    to bf16 of Z, M, dM and dZ on the way as well."""
    if case["op"].startswith("block"):
        return {"rel": 1.2e-2}
    return {"rel": 7e-3 if case["dtype"] == "bf16" else 1.2e-6}


def _fwht(a):
    """The unnormalised Walsh-Hadamard transform (Sylvester order) of every row of a [B, L] tensor."""
    B, L = a.shape
    h = 1
    while h < L:
        v = a.view(B, L // (2 * h), 2, h)
        a = torch.cat((v[:, :, :1] + v[:, :, 1:], v[:, :, :1] - v[:, :, 1:]), dim=2).view(B, L)
        h *= 2
    return a


def exact(case, seed):
    t = _inputs(case, seed)
    op, B, n, N, C = case["op"], case["B"], case["n"], case["N"], case["C"]
    L = N * C
    if op.startswith("sep"):
        g = (torch.exp(t["g_t"].double())[:, None] * torch.exp(t["g_c"].double())[None, :]).reshape(1, L)
    else:
        g = t["g"].double().reshape(1, L)

    def spectrum(a):           # of [B, n, C] planes, zero-padded to N tokens; orthonormal
        a = a.double().reshape(B, n * C)
        if n < N:
            a = torch.cat((a, a.new_zeros(B, (N - n) * C)), dim=1)
        return _fwht(a) / math.sqrt(L)

    def back(s):               # the inverse transform of [B, L] spectra, cropped to n tokens
        return (_fwht(s) / math.sqrt(L))[:, :n * C].reshape(B, n, C)

    z = t["x"].double()
    if op.startswith("block"):
        z = z @ t["w_in"].double().T
    sx = spectrum(z)
    mixed = back(sx * g)
    y = mixed @ t["w_out"].double().T if op.startswith("block") else mixed
    if not op.endswith("train"):
        return y
    dy = t["dy"].double()
    sd = spectrum(dy @ t["w_out"].double() if op == "block_train" else dy)
    dz = back(sd * g)
    dg = (sx * sd).sum(dim=0).view(N, C)
    if op == "mix_train":
        return {"y": y, "dx": dz, "dg": dg}
    if op == "sep_train":
        dlog = dg * g.view(N, C)
        return {"y": y, "dx": dz, "dg_t": dlog.sum(dim=1), "dg_c": dlog.sum(dim=0)}
    return {"y": y, "dx": dz @ t["w_in"].double(),
            "dw_in": dz.reshape(-1, C).T @ t["x"].double().reshape(-1, C), "dg": dg,
            "dw_out": dy.reshape(-1, C).T @ mixed.reshape(-1, C)}
