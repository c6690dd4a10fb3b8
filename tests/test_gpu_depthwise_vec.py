"""Small 3 x 3 depthwise layers of stride 2 (and any stride and dilation down the rows) and channel blocks of 64 against the oracle: one to a
few output columns per thread, channel counts around a thread's four."""
import pytest
import torch

from helpers import assert_within_bound, operand
from oracle import ref
from paper_2202_03293_b200 import binding as sg
from test_gpu_depthwise import run2d

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("N,Ho,Wo,C,st,dl", [(1, 1, 1, 4, (2, 2), (1, 1)), (2, 3, 2, 12, (2, 2), (1, 1)), (1, 7, 7, 24, (2, 2), (1, 1)), (3, 5, 3, 20, (1, 2), (2, 1)),
                                              (4, 4, 9, 64, (3, 2), (1, 1)), (2, 6, 5, 16, (1, 1), (1, 1)), (1, 13, 31, 100, (2, 2), (1, 1))])
def test_small_layers(N, Ho, Wo, C, st, dl, accumulate, dtype):
    O, want, S = run2d(N, Ho, Wo, C, 3, 3, st, dl, dtype, accumulate, extra=(1, 1))
    assert sg.sg_last_kernel_name() == "depthwise_vec_kernel"
    assert_within_bound(O, want, S, "depthwise, small")
    sg.sg_check()


# bf16 channel counts on both sides of the line between blocks of 64 and of 32
@pytest.mark.parametrize("C", [72, 96, 104, 136, 160, 200, 416])
@pytest.mark.parametrize("s,K", [(1, 3), (2, 3), (2, 5)])
def test_channel_blocks(C, s, K):
    O, want, S = run2d(30 if s == 1 else 9, 21, 27, C, K, K, (s, s), (1, 1), "bf16")       # (a tile per SM, or the kernel without tiles runs)
    assert sg.sg_last_kernel_name() == "depthwise_tma_kernel"
    assert_within_bound(O, want, S, "depthwise, channel blocks")
    sg.sg_check()


# bf16: numbers of thread blocks around one and two to an SM (shared memory keeps an SM to its share of them), tiles in their place from 7/3 on, and
# where tiles of 64 channels fill the rounds badly
@pytest.mark.parametrize("N,W,C,s,kernel", [(4, 14, 400, 1, "vec"), (4, 14, 408, 1, "vec"), (23, 14, 152, 1, "vec"), (24, 14, 152, 1, "vec"), (8, 28, 224, 1, "vec"),
                                            (24, 14, 264, 1, "tma"), (4, 14, 352, 2, "vec"), (4, 14, 416, 2, "vec"), (8, 28, 288, 1, "tma"), (24, 14, 224, 2, "tma")])
def test_lines(N, W, C, s, kernel):
    O, want, S = run2d(N, W, W, C, 3, 3, (s, s), (1, 1), "bf16")
    assert sg.sg_last_kernel_name() == f"depthwise_{kernel}_kernel"
    assert_within_bound(O, want, S, "depthwise, lines")
    sg.sg_check()


# f32: a lone block, a block more, one to an SM and one more (filters ahead of the multiplications on the outer sides)
@pytest.mark.parametrize("N,W,C", [(1, 7, 64), (2, 7, 64), (1, 30, 320), (1, 30, 628), (1, 30, 632), (7, 24, 184)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_filters_ahead(N, W, C, accumulate):
    O, want, S = run2d(N, W, W, C, 3, 3, (1, 1), (1, 1), "f32", accumulate)
    assert sg.sg_last_kernel_name() == "depthwise_vec_kernel"
    assert_within_bound(O, want, S, "depthwise, filters ahead")
    sg.sg_check()


# The kernel overlaps the launch ahead: its operands are the last thing that a long copy ahead writes, and a copy behind overwrites them, round after round.
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("N,W,C,s,K,kernel", [(2, 9, 24, 1, 3, "vec"), (1, 14, 200, 2, 3, "vec"), (3, 11, 36, 2, 2, "vec"), (16, 24, 64, 1, 5, "tma")])
def test_operands_of_the_launch_ahead(N, W, C, s, K, kernel, dtype):
    win = (W - 1) * s + K
    n_in, n_flt, cols, rounds = N * win * win * C, K * K * C, 4096, 6
    rows = 4096 + (n_in + n_flt + cols - 1) // cols
    start = rows * cols - n_in - n_flt
    buf = torch.empty(rows, cols, device="cuda", dtype=torch.float32 if dtype == "f32" else torch.bfloat16)
    I, F = buf.view(-1)[start:start + n_in].view(N, win, win, C), buf.view(-1)[start + n_in:].view(K, K, C)
    junk = torch.full_like(buf, 7.0)
    sources, outs, wants = [], [], []
    for r in range(rounds):
        a, i = operand((N, win, win, C), 9860, 2 * r, "normal", dtype)
        b, k = operand((K, K, C), 9860, 2 * r + 1, "normal", dtype)
        src = torch.zeros_like(buf)
        src.view(-1)[start:start + n_in], src.view(-1)[start + n_in:] = a.flatten(), b.flatten()
        sources.append(src)
        outs.append(torch.full((N, W, W, C), float("nan"), device="cuda"))
        wants.append(ref.depthwise_conv2d_nhwc_hwc(i, k, (s, s), (1, 1), out_hw=(W, W)))
    torch.cuda.synchronize()
    for src, O in zip(sources, outs):
        sg.sg_copy2d(src, buf)
        sg.sg_depthwise_conv2d_nhwc_hwc(I, F, O, (s, s), (1, 1))
        assert sg.sg_last_kernel_name() == f"depthwise_{kernel}_kernel"
        sg.sg_copy2d(junk, buf)
    torch.cuda.synchronize()
    for O, (want, S) in zip(outs, wants):
        assert_within_bound(O, want, S, "depthwise behind a copy")
    sg.sg_check()
