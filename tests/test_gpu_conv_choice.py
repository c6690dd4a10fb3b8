"""Unit-stride convolutions on both sides of the rule between strips and im2col, by the automatic choice and by the strip kernel,
against the oracle: one, three and five taps, channels that im2col pads and that it does not."""
import pytest
import torch

from helpers import assert_within_bound, operand
from oracle import ref
from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu
SEED = 9850


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("C", [32, 40, 64])
@pytest.mark.parametrize("KW,dl", [(1, 1), (3, 2), (5, 1)])
def test_strip_or_im2col(C, KW, dl, dtype):
    N, W, F = 37, 900, 32
    I, i = operand((N, W + (KW - 1) * dl, C), SEED, 1, "normal", dtype)
    K, k = operand((KW, C, F), SEED, 2, "normal", dtype)
    want, S = ref.conv1d_nwc_wcf(i, k, dilation=dl)
    strip = dtype == "bf16" or KW * C <= 192      # (a split filter beyond that does not stay in shared memory beside a strip)
    for kernel in (0, sg.SG_KERNEL_CONV_STRIP) if strip else (0,):
        O = torch.full((N, W, F), float("nan"), device="cuda")
        sg.sg_set_kernel_override(kernel)
        try:
            sg.sg_conv1d_nwc_wcf(I, K, O, 1, dl)
            torch.cuda.synchronize()
        finally:
            sg.sg_set_kernel_override(0)
        assert sg.sg_last_kernel_name() not in ("ffma_kernel", "")
        assert_within_bound(O, want, S, "strip or im2col")
    sg.sg_check()
