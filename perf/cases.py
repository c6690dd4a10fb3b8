"""Performance cases of the library: what a user's program has it do, through the public Python entry points.

A case is a dict of plain values.  Its "op" is one of
    matmul     C (+)= A.B on row-major operands
    linear     one training step of a linear layer: Y = relu(X.W + b), then dX = dY.W^T, dW += X^T.dY, db = column sums of dY
    conv1d     conv_1d_nwc_wcf      conv2d   conv_2d_nhwc_hwcf      depthwise   depthwise conv_2d_nhwc_hwc
    mem2d      the four memory-bound 2-D ops on one tensor: copy, transpose, column sums, row sums
Inputs are dense and drawn as in the benchmark: uniform[-1,1) for products and 1-D convolutions, N(0,1) for 2-D ones.
Outputs are f32 (copies and transposes: the input's type), allocated once and written by every pass.
"""
import math

import torch

from paper_2202_03293_b200 import binding as sg

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
BYTES = {"f32": 4, "bf16": 2}


def listed():
    return [
        # the smallest configured product: what a call costs when there is next to nothing to compute
        {"name": "matmul_128_f32", "op": "matmul", "dtype": "f32", "M": 128, "N": 128, "K": 128, "acc": False},
        # the corner of the configured sweep in f32: the framework's dominant kernel
        {"name": "matmul_4096_f32", "op": "matmul", "dtype": "f32", "M": 4096, "N": 4096, "K": 4096, "acc": False},
        # the largest configured product
        {"name": "matmul_8192_bf16", "op": "matmul", "dtype": "bf16", "M": 8192, "N": 8192, "K": 8192, "acc": False},
        # the configured skinny product: bound by reading A
        {"name": "matmul_skinny_bf16", "op": "matmul", "dtype": "bf16", "M": 16384, "N": 64, "K": 4096, "acc": False},
        # sizes that are multiples of nothing (counts of samples, classes, features): no row starts on a 16-byte boundary
        {"name": "matmul_odd_bf16", "op": "matmul", "dtype": "bf16", "M": 1531, "N": 1021, "K": 765, "acc": False},
        # forward and backward of a layer: fused bias + relu, both transposed layouts, an accumulated gradient
        {"name": "linear_4096x1024_f32", "op": "linear", "dtype": "f32", "T": 4096, "D": 1024, "F": 1024},
        # the configured 1-D convolution
        {"name": "conv1d_c3_f32", "op": "conv1d", "dtype": "f32", "N": 32, "W": 1024, "C": 64, "F": 128, "KW": 3, "s": 1, "d": 1},
        # the configured 2-D convolution
        {"name": "conv2d_c4_bf16", "op": "conv2d", "dtype": "bf16", "N": 16, "H": 56, "W": 56, "C": 64, "F": 128, "KH": 3, "KW": 3, "s": 1, "d": 1},
        # the paper's convolution constants (N,C,F,Kh,Kw) = (1,32,64,3,3) at stride 2, an odd image: one image, inference
        {"name": "conv2d_b1_s2_f32", "op": "conv2d", "dtype": "f32", "N": 1, "H": 55, "W": 55, "C": 32, "F": 64, "KH": 3, "KW": 3, "s": 2, "d": 1},
        # a MobileNet-like depthwise layer on a batch
        {"name": "depthwise_b32_bf16", "op": "depthwise", "dtype": "bf16", "N": 32, "H": 112, "W": 112, "C": 64, "K": 3, "s": 1},
        # the one size the paper names for the memory-bound ops, and one far beyond the caches
        {"name": "mem2d_250x960_f32", "op": "mem2d", "dtype": "f32", "R": 250, "C": 960},
        {"name": "mem2d_16384x12288_bf16", "op": "mem2d", "dtype": "bf16", "R": 16384, "C": 12288},
    ]


def _size(rng, lo, hi, step):
    """Log-uniform in [lo, hi], rounded down to a multiple of `step`."""
    v = int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))
    return max(step, v // step * step)


def _step(rng):
    """What sizes are multiples of: powers of two most of the time, anything in a third of the cases."""
    return rng.choice((64, 64, 8, 8, 1, 1))


def draw(rng):
    op = rng.choice(("matmul", "matmul", "matmul", "matmul", "linear", "linear", "conv1d", "conv2d", "conv2d", "depthwise", "mem2d", "mem2d"))
    dtype = rng.choice(("f32", "bf16"))
    # the most operations of a drawn case: the layouts that stay off the tensor cores are an order of magnitude slower
    most = 1.0e12 if dtype == "bf16" else 1.3e11
    while True:
        if op == "matmul":
            step = _step(rng)
            c = {"op": op, "dtype": dtype, "M": _size(rng, 64, 16384, step), "N": _size(rng, 64, 8192, step),
                 "K": _size(rng, 64, 8192, step), "acc": rng.random() < 0.25}
            limit = most if step % 8 == 0 else 4.0e9
        elif op == "linear":
            # feature counts are multiples of 8; the number of samples is anything
            step = rng.choice((64, 8))
            c = {"op": op, "dtype": dtype, "T": _size(rng, 64, 16384, 1), "D": _size(rng, 64, 4096, step), "F": _size(rng, 64, 4096, step)}
            limit = most / 4 if step == 64 else 1.2e9
        elif op == "conv1d":
            c = {"op": op, "dtype": dtype, "N": _size(rng, 1, 64, 1), "W": _size(rng, 50, 8192, 1), "C": rng.choice((16, 32, 40, 64, 80, 128, 256)),
                 "F": rng.choice((32, 64, 96, 128, 256)), "KW": rng.choice((1, 3, 3, 5, 7)), "s": rng.choice((1, 1, 2)), "d": rng.choice((1, 1, 1, 2))}
            limit = 2.0e10
        elif op == "conv2d":
            # 3 channels: the first layer of an image network
            c = {"op": op, "dtype": dtype, "N": _size(rng, 1, 64, 1), "H": 0, "W": _size(rng, 7, 112, 1), "C": rng.choice((3, 16, 32, 48, 64, 128, 256)),
                 "F": rng.choice((32, 64, 96, 128, 256)), "KH": 0, "KW": rng.choice((1, 3, 3, 3, 5)), "s": rng.choice((1, 1, 2)), "d": rng.choice((1, 1, 1, 2))}
            c["H"], c["KH"] = c["W"], c["KW"]
            limit = 2.0e10 if c["C"] > 3 else 4.0e9
        elif op == "depthwise":
            c = {"op": op, "dtype": dtype, "N": _size(rng, 1, 64, 1), "H": 0, "W": _size(rng, 7, 112, 1), "C": _size(rng, 16, 1024, 8),
                 "K": rng.choice((3, 3, 3, 5)), "s": rng.choice((1, 1, 2))}
            c["H"] = c["W"]
            limit = 2.0e9
        else:
            step = _step(rng)
            c = {"op": op, "dtype": dtype, "R": _size(rng, 64, 16384, step), "C": _size(rng, 64, 16384, step)}
            limit = 2.5e8
        if work(c)["flops"] <= limit:
            return c


def _rand(gen, shape, dtype, normal=False):
    if normal:
        return torch.randn(shape, generator=gen, device="cuda").to(DTYPES[dtype])
    return torch.rand(shape, generator=gen, device="cuda").mul_(2).sub_(1).to(DTYPES[dtype])


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    op, dt = case["op"], case["dtype"]
    out = dict(device="cuda", dtype=torch.float32)
    s = {"case": case}
    if op == "matmul":
        s["A"], s["B"] = _rand(gen, (case["M"], case["K"]), dt), _rand(gen, (case["K"], case["N"]), dt)
        s["C"] = torch.zeros(case["M"], case["N"], **out)
    elif op == "linear":
        T, D, F = case["T"], case["D"], case["F"]
        s["X"], s["W"], s["dY"] = _rand(gen, (T, D), dt), _rand(gen, (D, F), dt), _rand(gen, (T, F), dt)
        s["b"] = _rand(gen, (F,), "f32")
        s["Y"], s["dX"], s["dW"], s["db"] = torch.zeros(T, F, **out), torch.zeros(T, D, **out), torch.zeros(D, F, **out), torch.zeros(F, **out)
    elif op == "conv1d":
        w_in = (case["W"] - 1) * case["s"] + (case["KW"] - 1) * case["d"] + 1
        s["I"], s["K"] = _rand(gen, (case["N"], w_in, case["C"]), dt), _rand(gen, (case["KW"], case["C"], case["F"]), dt)
        s["O"] = torch.zeros(case["N"], case["W"], case["F"], **out)
    elif op == "conv2d":
        h_in, w_in = ((case[e] - 1) * case["s"] + (case["K" + e] - 1) * case["d"] + 1 for e in ("H", "W"))
        s["I"] = _rand(gen, (case["N"], h_in, w_in, case["C"]), dt, True)
        s["K"] = _rand(gen, (case["KH"], case["KW"], case["C"], case["F"]), dt, True)
        s["O"] = torch.zeros(case["N"], case["H"], case["W"], case["F"], **out)
    elif op == "depthwise":
        h_in, w_in = ((case[e] - 1) * case["s"] + case["K"] for e in ("H", "W"))
        s["I"], s["K"] = _rand(gen, (case["N"], h_in, w_in, case["C"]), dt, True), _rand(gen, (case["K"], case["K"], case["C"]), dt, True)
        s["O"] = torch.zeros(case["N"], case["H"], case["W"], case["C"], **out)
    else:
        R, C = case["R"], case["C"]
        s["A"] = _rand(gen, (R, C), dt)
        s["copy"], s["t"] = torch.zeros(R, C, device="cuda", dtype=DTYPES[dt]), torch.zeros(C, R, device="cuda", dtype=DTYPES[dt])
        s["col"], s["row"] = torch.zeros(C, **out), torch.zeros(R, **out)
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "matmul":
        return sg.sg_matmul(s["A"], s["B"], s["C"], sg.SG_ACCUMULATE if case["acc"] else sg.SG_OVERWRITE)
    if op == "linear":
        X, W, dY = s["X"], s["W"], s["dY"]
        return (sg.sg_matmul_bias_act(X, W, s["b"], s["Y"], sg.SG_ACT_RELU),
                sg.sg_matmul(dY, W.t(), s["dX"]),
                sg.sg_matmul(X.t(), dY, s["dW"], sg.SG_ACCUMULATE),
                sg.sg_colred2d(dY, s["db"]))
    if op == "conv1d":
        return sg.sg_conv1d_nwc_wcf(s["I"], s["K"], s["O"], case["s"], case["d"])
    if op == "conv2d":
        return sg.sg_conv2d_nhwc_hwcf(s["I"], s["K"], s["O"], (case["s"], case["s"]), (case["d"], case["d"]))
    if op == "depthwise":
        return sg.sg_depthwise_conv2d_nhwc_hwc(s["I"], s["K"], s["O"], (case["s"], case["s"]))
    A = s["A"]
    return (sg.sg_copy2d(A, s["copy"]), sg.sg_transpose2d(A, s["t"]), sg.sg_colred2d(A, s["col"]), sg.sg_rowred2d(A, s["row"]))


def work(case):
    """Bytes (each operand of each call once; an accumulated output is read and written) and operations of one pass."""
    op, es = case["op"], BYTES[case["dtype"]]
    if op == "matmul":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": (M * K + K * N) * es + M * N * (8 if case["acc"] else 4), "flops": 2 * M * N * K}
    if op == "linear":
        T, D, F = case["T"], case["D"], case["F"]
        return {"bytes": (2 * T * D + 2 * D * F + 3 * T * F) * es + (T * F + T * D + 2 * D * F + 2 * F) * 4, "flops": 6 * T * D * F + T * F}
    if op in ("conv1d", "conv2d"):
        H, KH = case.get("H", 1), case.get("KH", 1)
        h_in, w_in = (H - 1) * case["s"] + (KH - 1) * case["d"] + 1, (case["W"] - 1) * case["s"] + (case["KW"] - 1) * case["d"] + 1
        outs = case["N"] * H * case["W"] * case["F"]
        taps = KH * case["KW"] * case["C"]
        # a stride that skips pixels (1-wide windows) leaves them unread
        read = case["N"] * case["C"] * (H if KH == 1 else h_in) * (case["W"] if case["KW"] == 1 else w_in)
        return {"bytes": (read + taps * case["F"]) * es + outs * 4, "flops": 2 * outs * taps}
    if op == "depthwise":
        h_in, w_in = (case["H"] - 1) * case["s"] + case["K"], (case["W"] - 1) * case["s"] + case["K"]
        outs = case["N"] * case["H"] * case["W"] * case["C"]
        return {"bytes": (case["N"] * h_in * w_in + case["K"] ** 2) * case["C"] * es + outs * 4, "flops": 2 * outs * case["K"] ** 2}
    R, C = case["R"], case["C"]
    return {"bytes": 6 * R * C * es + (R + C) * 4, "flops": 2 * R * C}


def tolerance(case):
    """Sums in f32: about 1e-5, and more for long reductions, where accumulators that round towards zero (the tensor
    cores' do) drift in proportion to the number of terms.  Copies and transposes are in the same answer as their
    sums; they move bits."""
    op = case["op"]
    if op == "matmul":
        terms = case["K"]
    elif op == "linear":
        terms = max(case["T"], case["D"], case["F"])
    else:
        terms = 0
    return {"rel": max(1e-5, 6e-9 * terms)}
