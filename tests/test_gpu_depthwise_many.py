"""Tiled depthwise convolutions with so many tiles that several times as many thread blocks as fit the chip share them: one and
three channel blocks of 64, blocks of 32 that miss channels, uneven shares, stride 2, accumulation."""
import pytest
import torch

from helpers import assert_within_bound, operand
from oracle import ref
from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu
SEED = 9950


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("N,H,W,C,st,accumulate", [(33, 112, 112, 64, 1, False), (13, 112, 105, 192, 1, True), (40, 97, 97, 72, 1, False),
                                                   (100, 71, 97, 24, 1, True), (24, 131, 123, 128, 2, False), (13, 112, 113, 200, 1, False)])
def test_many_tiles(N, H, W, C, st, accumulate, dtype):
    Ho, Wo = (H - 3) // st + 1, (W - 3) // st + 1
    I, i = operand((N, H, W, C), SEED, 1, "normal", dtype)
    F, f = operand((3, 3, C), SEED, 2, "normal", dtype)
    O = torch.full((N, Ho, Wo, C), 1.0 if accumulate else float("nan"), device="cuda")
    sg.sg_depthwise_conv2d_nhwc_hwc(I, F, O, (st, st), (1, 1), sg.SG_ACCUMULATE if accumulate else sg.SG_OVERWRITE)
    torch.cuda.synchronize()
    sg.sg_check()
    assert sg.sg_last_kernel_name() == "depthwise_tma_kernel"
    want, S = ref.depthwise_conv2d_nhwc_hwc(i, f, (st, st), (1, 1))
    assert_within_bound(O, want + accumulate, S + accumulate, "depthwise, many tiles")
