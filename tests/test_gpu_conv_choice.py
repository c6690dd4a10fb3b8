"""Unit-stride convolutions on both sides of the rules between strips, im2col, the filter as the M operand and the kernel for small problems, against
the oracle: one, three and five taps, channels that im2col pads and that it does not, outputs that are one matrix and padded ones."""
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
@pytest.mark.parametrize("pad", [0, 1])
def test_strip_or_im2col(C, KW, dl, pad, dtype):
    N, W, F = 37, 900, 32
    I, i = operand((N, W + (KW - 1) * dl, C), SEED, 1, "normal", dtype)
    K, k = operand((KW, C, F), SEED, 2, "normal", dtype)
    want, S = ref.conv1d_nwc_wcf(i, k, dilation=dl)
    fits = dtype == "bf16" or KW * C <= 192      # (a split filter beyond that does not stay in shared memory beside a strip)
    strips = pad == 1 or (dtype == "bf16" and KW >= (3 if C % 64 else 5))
    chosen = "conv_strip_kernel" if strips and fits else "gather_gemm_kernel" if pad else "tc_gemm_kernel"
    for kernel in (0, sg.SG_KERNEL_CONV_STRIP) if fits else (0,):
        wide = torch.full((N, W + 2 * pad, F), float("nan"), device="cuda")
        O = wide[:, pad:pad + W]
        sg.sg_set_kernel_override(kernel)
        try:
            sg.sg_conv1d_nwc_wcf(I, K, O, 1, dl)
            torch.cuda.synchronize()
        finally:
            sg.sg_set_kernel_override(0)
        assert sg.sg_last_kernel_name() == f"{'conv_strip_kernel' if kernel else chosen}<{dtype}>"
        assert_within_bound(O, want, S, "strip or im2col")
        assert int(torch.isnan(wide).sum()) == 2 * pad * N * F
    sg.sg_check()


# Convolutions into padded outputs, which the im2col kernel does not take.  Where a filter stays or streams past the runs of input rows, the kernel for small problems
# has that kernel to beat; elsewhere (strides) the gather kernel.
@pytest.mark.parametrize("N,W,C,F,KW,s,dtype,kernel", [
    (1, 77, 64, 128, 3, 1, "bf16", "conv_wide_kernel"), (4, 32, 64, 128, 3, 1, "bf16", "conv_wide_kernel"), (27, 24, 48, 64, 1, 1, "f32", "conv_strip_kernel"),
    (3, 10, 16, 96, 3, 1, "bf16", "small_gemm_kernel"), (14, 9, 40, 64, 1, 1, "f32", "small_gemm_kernel"), (6, 10, 64, 96, 3, 2, "f32", "small_gemm_kernel"),
    (16, 31, 16, 64, 3, 2, "f32", "gather_gemm_kernel"), (24, 40, 64, 96, 3, 2, "bf16", "gather_gemm_kernel")])
def test_padded_outputs(N, W, C, F, KW, s, dtype, kernel):
    win = (W - 1) * s + KW
    I, i = operand((N, win, win, C), SEED, 3, "normal", dtype)
    K, k = operand((KW, KW, C, F), SEED, 4, "normal", dtype)
    wide = torch.full((N, W + 2, W + 2, F), float("nan"), device="cuda")
    O = wide[:, 1:-1, 1:-1]
    sg.sg_conv2d_nhwc_hwcf(I, K, O, (s, s))
    torch.cuda.synchronize()
    assert sg.sg_last_kernel_name() == f"{kernel}<{dtype}>"
    want, S = ref.conv2d_nhwc_hwcf(i, k, (s, s))
    assert_within_bound(O, want, S, "padded output")
    assert int(torch.isnan(wide).sum()) == wide.numel() - O.numel()
    sg.sg_check()


# f32, im2col or the filter as the M operand: a long reduction over few positions, filters that stream past many, filters that stay
@pytest.mark.parametrize("N,W,C,F,KW,kernel", [(8, 28, 256, 256, 3, "tc_gemm_kernel"), (10, 57, 16, 128, 3, "conv_wide_kernel"), (5, 80, 16, 128, 3, "conv_wide_kernel"),
                                               (18, 47, 16, 64, 3, "tc_gemm_kernel")])
def test_wide_or_im2col(N, W, C, F, KW, kernel):
    I, i = operand((N, W + KW - 1, W + KW - 1, C), SEED, 5, "normal", "f32")
    K, k = operand((KW, KW, C, F), SEED, 6, "normal", "f32")
    O = torch.full((N, W, W, F), float("nan"), device="cuda")
    sg.sg_conv2d_nhwc_hwcf(I, K, O)
    torch.cuda.synchronize()
    assert sg.sg_last_kernel_name() == f"{kernel}<f32>"
    want, S = ref.conv2d_nhwc_hwcf(i, k)
    assert assert_within_bound(O, want, S, "wide or im2col") < 4e-6
    sg.sg_check()


# few positions and a long reduction: the im2col kernel deals it out over the SMs; many positions, or few filters that stay: the filter as the M operand
@pytest.mark.parametrize("N,H,C,KH,F,kernel", [(5, 15, 128, 5, 96, "tc_gemm_kernel<bf16>"), (1, 31, 256, 3, 64, "tc_gemm_kernel<bf16>"), (16, 56, 64, 3, 128, "conv_wide_kernel<bf16>"), (29, 37, 32, 5, 32, "conv_wide_kernel<bf16>")])
def test_im2col_or_filter_as_the_m_operand(N, H, C, KH, F, kernel):
    I, i = operand((N, H + KH - 1, H + KH - 1, C), SEED, 31, "normal", "bf16")
    K, k = operand((KH, KH, C, F), SEED, 32, "normal", "bf16")
    O = torch.full((N, H, H, F), float("nan"), device="cuda")
    sg.sg_conv2d_nhwc_hwcf(I, K, O)
    torch.cuda.synchronize()
    assert sg.sg_last_kernel_name() == kernel
    want = torch.nn.functional.conv2d(I[:2].double().permute(0, 3, 1, 2), K.double().permute(3, 2, 0, 1)).permute(0, 2, 3, 1)
    S = torch.nn.functional.conv2d(I[:2].double().abs().permute(0, 3, 1, 2), K.double().abs().permute(3, 2, 0, 1)).permute(0, 2, 3, 1)
    assert ((O[:2].double() - want).abs() <= 4e-6 * S).all()      # the truncating sum of up to 3200 products
    sg.sg_check()
