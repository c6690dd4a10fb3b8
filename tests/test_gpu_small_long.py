"""bf16 on the kernel for small problems: reductions of more than 2048 products, with partial sums as short as those of the gather kernel, which would run them
otherwise, and short reductions of many tiles, three thread blocks to an SM."""
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


# bf16, up to three stages of 128 and more than two tiles of 32 x 32 per SM: three thread blocks to an SM; one stage more, a tile row fewer
@pytest.mark.parametrize("M,N,K", [(9504, 32, 384), (9472, 32, 384), (4800, 72, 16), (9504, 32, 392), (3000, 168, 104)])
@pytest.mark.parametrize("a_t,b_t", [(False, False), (True, False), (False, True), (True, True)])
def test_three_blocks_to_an_sm(M, N, K, a_t, b_t):
    g = torch.Generator(device="cuda").manual_seed(9960)
    A = (torch.rand(*((K, M) if a_t else (M, K)), generator=g, device="cuda") * 2 - 1).bfloat16()
    B = (torch.rand(*((N, K) if b_t else (K, N)), generator=g, device="cuda") * 2 - 1).bfloat16()
    A, B = A.t() if a_t else A, B.t() if b_t else B
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_matmul(A, B, C)
    torch.cuda.synchronize()
    err = (C.double() - A.double() @ B.double()).abs()
    # at most 48 truncating additions of a warp and 8 sums: 56 * 2^-23
    assert (err <= 7e-6 * (A.double().abs() @ B.double().abs())).all()
    sg.sg_check()


@pytest.mark.parametrize("W,C,s", [(97, 40, 1), (97, 24, 2), (96, 16, 1)])
def test_three_blocks_to_an_sm_on_convolutions(W, C, s):
    g = torch.Generator(device="cuda").manual_seed(9961)
    win = (W - 1) * s + 3
    I = torch.randn(1, win, win, C, generator=g, device="cuda").bfloat16()
    K = torch.randn(3, 3, C, 40, generator=g, device="cuda").bfloat16()
    O = torch.full((1, W + 1, W + 1, 40), float("nan"), device="cuda")[:, :W, :W]
    sg.sg_conv2d_nhwc_hwcf(I, K, O, (s, s))
    torch.cuda.synchronize()
    want = torch.nn.functional.conv2d(I.double().permute(0, 3, 1, 2), K.double().permute(3, 2, 0, 1), stride=s).permute(0, 2, 3, 1)
    bound = torch.nn.functional.conv2d(I.double().abs().permute(0, 3, 1, 2), K.double().abs().permute(3, 2, 0, 1), stride=s).permute(0, 2, 3, 1)
    assert ((O.double() - want).abs() <= 7e-6 * bound).all()
    sg.sg_check()
