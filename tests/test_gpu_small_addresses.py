"""Addresses of the kernel for small problems: extents of one, channel counts that divide nothing, filters with gaps, images with gaps,
against the oracle."""
import pytest
import torch

from helpers import assert_within_bound, operand
from oracle import ref
from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu
SEED = 9800


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("N,Ho,Wo,C,F,KH,KW,s,d", [(5, 1, 1, 24, 40, 3, 3, 1, 1), (3, 7, 1, 40, 32, 1, 5, 2, 1), (2, 1, 9, 72, 40, 5, 1, 1, 2),
                                                    (1, 13, 11, 8, 72, 3, 7, 3, 2), (1, 6, 5, 136, 32, 3, 3, 2, 1)])
@pytest.mark.parametrize("gap", [0, 8])
def test_convolutions(N, Ho, Wo, C, F, KH, KW, s, d, gap, dtype):
    hin, win = (Ho - 1) * s + (KH - 1) * d + 1, (Wo - 1) * s + (KW - 1) * d + 1
    I, i = operand((N, hin, win, C), SEED, 1, "normal", dtype)
    K, k = operand((KH, KW, C, F), SEED, 2, "normal", dtype)
    if gap:      # pixels and filter taps further apart than their extents
        wide_i, wide_k = torch.zeros(N, hin, win + 1, C + gap, device="cuda", dtype=I.dtype), torch.zeros(KH, KW + 1, C + gap, F, device="cuda", dtype=K.dtype)
        wide_i[:, :, :win, :C], wide_k[:, :KW, :C] = I, K
        I, K = wide_i[:, :, :win, :C], wide_k[:, :KW, :C]
    O = torch.full((N, Ho, Wo, F), float("nan"), device="cuda")
    sg.sg_conv2d_nhwc_hwcf(I, K, O, (s, s), (d, d))
    torch.cuda.synchronize()
    assert sg.sg_last_kernel_name() == f"small_gemm_kernel<{dtype}>"
    want, S = ref.conv2d_nhwc_hwcf(i, k, (s, s), (d, d), out_hw=(Ho, Wo))
    assert assert_within_bound(O, want, S, "small convolution") < 4e-6
    sg.sg_check()
