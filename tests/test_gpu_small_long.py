"""bf16 reductions of more than 2048 products on the kernel for small problems: partial sums as short as the gather kernel's, which would run them otherwise."""
import pytest
import torch

from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu


def relative(O, want):
    return float((O.double() - want).norm() / want.norm())


# one image of 6 x 6 outputs, 5 x 5 windows: 2000 (one accumulator a warp), 2200, 3000 and 4000 products of positive values
@pytest.mark.parametrize("C", [80, 88, 120, 160])
@pytest.mark.parametrize("s", [1, 2])
def test_error_of_long_sums(C, s):
    g = torch.Generator(device="cuda").manual_seed(9950)
    win = 5 * s + 5
    I = torch.rand(1, win, win, C, generator=g, device="cuda").bfloat16()
    K = torch.rand(5, 5, C, 64, generator=g, device="cuda").bfloat16()
    want = torch.nn.functional.conv2d(I.double().permute(0, 3, 1, 2), K.double().permute(3, 2, 0, 1), stride=s).permute(0, 2, 3, 1)
    err = {}
    for family in (sg.SG_KERNEL_AUTO, sg.SG_KERNEL_TENSOR):
        O = torch.full((1, 6, 6, 64), float("nan"), device="cuda")
        sg.sg_set_kernel_override(family)
        try:
            sg.sg_conv2d_nhwc_hwcf(I, K, O, (s, s))
            torch.cuda.synchronize()
        finally:
            sg.sg_set_kernel_override(sg.SG_KERNEL_AUTO)
        err[sg.sg_last_kernel_name()] = relative(O, want)
    assert set(err) == {"small_gemm_kernel<bf16>", "gather_gemm_kernel<bf16>"}
    # 256 truncating additions drift by about 256 * 2^-25 of the sum of a chunk, which is up to the whole of a warp's share: 3.1e-7 measured for 2048 and more
    assert err["small_gemm_kernel<bf16>"] < 4e-7, err
    sg.sg_check()
