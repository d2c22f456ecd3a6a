"""The convolution work whose speed this repository watches.

A case is one layer (sizes and stride), the way a program takes it through the library (``op``) and the
tensor-core mode.  The listed cases are layers of ``paper_2306_14320_b200.workloads`` at the batch sizes 1, 32
and 128 that the benchmark sweeps, plus one general shape; ``draw`` gives further ones of the same ranges.

``op``, in the words of include/im2win.h:
  conv         im2win_conv on the untransformed input: Algorithm 1, then Algorithm 2 (the paper's call)
  fused        im2win_conv with IM2WIN_SRC_NCHW_FUSED: the same result without an im2win tensor in memory
  im2win       im2win_transform, then im2win_conv on the tensor it wrote (a program that keeps the tensor)
  im2win_bf16  im2win_transform_bf16, then im2win_conv on the bf16 tensor
  transform    im2win_transform alone
  nhwc         im2win_conv_nhwc, fused source: channels-last output for a consumer that wants it
"""
from __future__ import annotations

import math

import torch

from paper_2306_14320_b200 import binding as b

MODES = {"tf32": b.MODE_TF32, "bf16": b.MODE_BF16}


def _case(name, op, mode, N, C, H, W, K, Fh, Fw, s, pad):
    return {"name": name, "op": op, "mode": mode, "N": N, "C": C, "H": H, "W": W, "K": K, "Fh": Fh, "Fw": Fw,
            "stride": s, "pad": pad}


def listed():
    return [
        # The smallest call: one 32x32 image, a few thousand outputs.  Launches and host work are all of it.
        _case("tiny_b1", "conv", "tf32", 1, 3, 32, 32, 16, 3, 3, 1, 0),
        # One image through a deep layer: the latency of single-image inference (a long reduction, few outputs).
        _case("deep3x3_b1", "fused", "bf16", 1, 256, 16, 16, 256, 3, 3, 1, 1),
        # One image through the entry layer of a residual network.
        _case("stem7x7_b1", "conv", "tf32", 1, 3, 230, 230, 64, 7, 7, 2, 3),
        # The headline layer of the benchmark, whole batch, the paper's transform + convolution in TF32.
        _case("resnet3x3", "conv", "tf32", 128, 64, 58, 58, 64, 3, 3, 1, 1),
        # The same layer as a serving batch runs it: fused, BF16.
        _case("resnet3x3_b32", "fused", "bf16", 32, 64, 58, 58, 64, 3, 3, 1, 1),
        # Stride-2 downsampling between two stages, fused, TF32.
        _case("down3x3", "fused", "tf32", 128, 128, 58, 58, 256, 3, 3, 2, 1),
        # Last stage of a residual network: many channels, 7x7 outputs, the im2win tensor kept by the caller.
        _case("sweep_L12", "im2win", "bf16", 128, 512, 9, 9, 512, 3, 3, 1, 1),
        # Odd image side (15), 384 filters, a serving batch, TF32.
        _case("sweep_L4_b32", "conv", "tf32", 32, 384, 15, 15, 384, 3, 3, 1, 1),
        # 5x5 layer with the im2win tensor stored as bf16 (half the workspace).
        _case("sweep_L2", "im2win_bf16", "bf16", 128, 96, 31, 31, 256, 5, 5, 1, 2),
        # The transform alone on an 11x11 stride-4 stem with an odd row length (227).
        _case("sweep_L1", "transform", "tf32", 128, 3, 227, 227, 96, 11, 11, 4, 0),
        # A general shape: rectangular filter, channel and filter counts that no tile divides, a channels-last output.
        _case("general_3x5", "nhwc", "bf16", 16, 40, 45, 61, 72, 3, 5, 1, 0),
        # The largest: a wide early layer, 228 GFLOP and 1.2 GB of input and output, fused, TF32.
        _case("table1_Conv8", "fused", "tf32", 128, 64, 112, 112, 128, 3, 3, 1, 0),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _count(rng, lo, hi):
    """A channel or filter count: usually a multiple of 32 or 16, as network layers have, else any number."""
    n = _log_int(rng, lo, hi)
    r = rng.random()
    m = 32 if r < 0.5 else (16 if r < 0.75 else 1)
    return max(lo, min(hi, (n + m // 2) // m * m))


def draw(rng):
    """One more case: filter family, layer sizes, batch (1 to 128, over its logarithm), call and mode, none of
    it larger than the largest listed case."""
    while True:
        family = rng.choice(("3x3", "3x3", "3x3", "3x3s2", "5x5", "stem", "rect"))
        pad_wanted = rng.random() < 0.6
        if family == "stem":
            C = 3
            Fh = Fw = rng.choice((7, 11, 3))
            s = {7: 2, 11: 4, 3: 1}[Fh]
            H = W = _log_int(rng, 64, 231)
            K = _count(rng, 16, 96)
        elif family == "rect":
            Fh, Fw, s = rng.choice(((1, 1, 1), (1, 3, 1), (3, 1, 1), (1, 7, 1), (7, 1, 1), (3, 5, 1), (5, 3, 1),
                                    (2, 2, 2), (4, 4, 2), (3, 4, 1)))
            C, K = _count(rng, 16, 256), _count(rng, 16, 384)
            H, W = _log_int(rng, 10, 64), _log_int(rng, 10, 64)
        elif family == "5x5":
            Fh = Fw = 5
            s = 1
            C, K = _count(rng, 16, 128), _count(rng, 32, 256)
            H = W = _log_int(rng, 12, 48)
        else:
            Fh = Fw = 3
            s = 2 if family == "3x3s2" else 1
            C, K = _count(rng, 16, 512), _count(rng, 16, 512)
            H = _log_int(rng, 7, 112)
            W = H if rng.random() < 0.7 else _log_int(rng, 7, 112)
        N = _log_int(rng, 1, 128)
        mode = rng.choice(("tf32", "bf16"))
        op = rng.choice(("conv", "conv", "fused", "fused", "im2win", "im2win_bf16", "transform", "nhwc"))
        if op == "transform":
            mode = "tf32"  # (the fp32 tensor, which either mode can consume)
        if op == "im2win_bf16":
            mode = "bf16"
            if not (s == 1 and Fh == Fw and Fh in (3, 5) and C % 32 == 0):
                continue  # (the library takes a bf16 tensor for these filters and channel counts)
        pad = min(Fh // 2, Fw // 2) if pad_wanted else 0
        c = _case("", op, mode, N, C, H, W, K, Fh, Fw, s, pad if min(H, W) > 4 * pad else 0)
        del c["name"]
        w, top = work(c), work(listed()[-1])
        if max(w["flops"] / top["flops"], w["bytes"] / top["bytes"]) <= 0.9:
            return c


def _dims(c):
    return (c["N"], c["C"], c["H"], c["W"], c["K"], c["Fh"], c["Fw"], c["stride"])


def _out_dims(c):
    return (c["H"] - c["Fh"]) // c["stride"] + 1, (c["W"] - c["Fw"]) // c["stride"] + 1


def _inputs(case, seed):
    """N(0,1) values inside an explicit zero ring of `pad`; Kaiming-normal filters (none for the transform)."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    N, C, H, W, K, Fh, Fw, _ = _dims(case)
    p = case["pad"]
    x = torch.zeros((N, C, H, W), device=dev)
    x[:, :, p:H - p, p:W - p].normal_(generator=gen)
    if case["op"] == "transform":
        return x, None
    return x, torch.empty((K, C, Fh, Fw), device=dev).normal_(generator=gen) * math.sqrt(2.0 / (C * Fh * Fw))


def prepare(case, seed):
    dev = torch.device("cuda")
    N, C, H, W, K, Fh, Fw, _ = dims = _dims(case)
    Ho, Wo = _out_dims(case)
    op, mode = case["op"], MODES[case["mode"]]
    x, f = _inputs(case, seed)
    st = {"op": op, "mode": mode, "dims": dims, "x": x}
    if op in ("transform", "im2win"):
        st["xhat"] = torch.empty((N, C, Ho, W * Fh), device=dev)
    elif op == "im2win_bf16":
        st["xhat"] = torch.empty((N, C, Ho, W * Fh), device=dev, dtype=torch.bfloat16)
    if op == "transform":
        return st
    st["f"] = f
    st["out"] = torch.empty((N, Ho, Wo, K) if op == "nhwc" else (N, K, Ho, Wo), device=dev)
    # The workspace with which the fastest kernels apply; the fused calls get what the unfused call would want,
    # so that shapes without a fused kernel are served too.
    kind = {"im2win": b.SRC_IM2WIN, "im2win_bf16": b.SRC_IM2WIN_BF16}.get(op, b.SRC_NCHW)
    nbytes = b.conv_workspace_bytes(dims, kind, mode)
    if op in ("fused", "nhwc"):
        nbytes = max(nbytes, b.conv_workspace_bytes(dims, b.SRC_NCHW_FUSED, mode))
    st["ws"] = torch.empty(nbytes, device=dev, dtype=torch.uint8) if nbytes else None
    if op == "conv":  # the call leaves the im2win tensor at the start of the workspace
        st["xhat"] = st["ws"][:4 * N * C * Ho * W * Fh].view(torch.float32)
    return st


def run(st):
    op, dims = st["op"], st["dims"]
    if op == "transform":
        b.transform(st["x"], dims, st["xhat"])
        return st["xhat"]
    f, mode, out, ws = st["f"], st["mode"], st["out"], st["ws"]
    if op == "conv":
        b.conv(st["x"], b.SRC_NCHW, f, dims, mode, out, ws)
        return out, st["xhat"]
    if op == "fused":
        b.conv(st["x"], b.SRC_NCHW_FUSED, f, dims, mode, out, ws)
        return out
    if op == "nhwc":
        b.conv_nhwc(st["x"], b.SRC_NCHW_FUSED, f, dims, mode, out, ws)
        return out
    if op == "im2win":
        b.transform(st["x"], dims, st["xhat"])
        b.conv(st["xhat"], b.SRC_IM2WIN, f, dims, mode, out, ws)
        return out, st["xhat"]
    b.transform_bf16(st["x"], dims, st["xhat"])
    b.conv(st["xhat"], b.SRC_IM2WIN_BF16, f, dims, mode, out, ws)
    return out, st["xhat"]


def exact(case, seed):
    """What run() returns, in 64 bits: the im2win tensor is a copy of input elements (rounded to bf16 where it is
    stored so), the convolution Eq. 1 as one matrix product per image."""
    N, C, H, W, K, Fh, Fw, s = _dims(case)
    Ho, Wo = _out_dims(case)
    op = case["op"]
    x, f = _inputs(case, seed)
    xhat = None
    if op in ("transform", "conv", "im2win", "im2win_bf16"):  # Ihat[i][r][m][k*Fh+u] = I[i][r][m*s+u][k]
        xhat = torch.empty((N, C, Ho, W, Fh), device=x.device)
        for u in range(Fh):
            xhat[..., u] = x[:, :, u:u + (Ho - 1) * s + 1:s]
        xhat = xhat.view(N, C, Ho, W * Fh)
        if op == "transform":
            return xhat
        if op == "im2win_bf16":
            xhat = xhat.bfloat16()
        if op == "conv":
            xhat = xhat.view(-1)
    f64 = f.double().view(K, C * Fh * Fw)
    out = torch.empty((N, K, Ho * Wo), device=x.device, dtype=torch.float64)
    for i in range(N):
        cols = torch.nn.functional.unfold(x[i:i + 1].double(), (Fh, Fw), stride=s)[0]
        torch.mm(f64, cols, out=out[i])
    out = out.view(N, K, Ho, Wo)
    if op == "nhwc":
        return out.permute(0, 2, 3, 1).contiguous()
    return out if op == "fused" else (out, xhat)


def work(case):
    """Multiplications and additions of Eq. 1; bytes: the input rows and the filter read once, the output and,
    where the call leaves it to the caller, the im2win tensor written once (and read once by a convolution that
    is called on it)."""
    N, C, H, W, K, Fh, Fw, s = _dims(case)
    Ho, Wo = _out_dims(case)
    op = case["op"]
    win = N * C * Ho * W * Fh * (2 if op == "im2win_bf16" else 4)
    nbytes = 4 * N * C * min(H, (Ho - 1) * s + Fh) * W
    if op in ("transform", "conv"):
        nbytes += win
    elif op in ("im2win", "im2win_bf16"):
        nbytes += 2 * win
    if op == "transform":
        return {"bytes": nbytes, "flops": 0}
    nbytes += 4 * K * C * Fh * Fw + 4 * N * K * Ho * Wo
    return {"bytes": nbytes, "flops": 2 * N * K * Ho * Wo * C * Fh * Fw}


def tolerance(case):
    """The transform copies.  The convolution's operands are TF32 (the low 13 mantissa bits unread) or bf16,
    products and sums fp32: against a sum of the same fp32 values in 64 bits the listed and ten drawn cases
    are off by 7.6e-4 to 8.0e-4 in norm and 2.3e-3 at the largest difference (TF32), 2.4e-3 and 1.3e-2 (bf16).
    Stated: four times that."""
    if case["op"] == "transform":
        return "exact"
    return {"rel": 1e-2, "max": 5e-2} if case["mode"] == "bf16" else {"rel": 3e-3, "max": 1e-2}
