"""The CUDA-core kernel's 32 x 32 tiles, which run by themselves where an unaligned problem is small: edges of tiles, of a fetch of 128 k and of its
threads along k, either operand contiguous along either index or along none, against the oracle."""
import numpy as np
import pytest
import torch

from helpers import assert_within_bound, operand
from oracle import ref
from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu
SEED = 9800


def strided(t, order):
    """The same values stored row by row, column by column, or with gaps everywhere."""
    if order == "t":
        return t.t().contiguous().t()
    if order == "gaps":
        out = torch.empty(t.shape[0] * 3 + 1, t.shape[1] * 2 + 1, dtype=t.dtype, device=t.device)[1::3, 1::2]
        return out.copy_(t)
    return t


# one k to a fetch's whole and one more, tiles of one row or column, the last of 31 and the first of 33
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("orders", [("n", "n"), ("t", "t"), ("gaps", "n"), ("t", "gaps")])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (31, 33, 32), (33, 31, 33), (65, 7, 64), (97, 65, 65), (127, 127, 128), (5, 95, 129), (63, 1, 385), (1025, 33, 27)])
def test_products(M, N, K, orders, dtype):
    A, a = operand((M, K), SEED, 1, "uniform", dtype)
    B, b = operand((K, N), SEED, 2, "uniform", dtype)
    A, B = strided(A, orders[0]), strided(B, orders[1])
    want, S = ref.matmul(a, b)
    wide = torch.full((M, 2 * N + 1), float("nan"), device="cuda")
    for C in (torch.full((M, N), float("nan"), device="cuda"), wide[:, 1::2]):
        sg.sg_matmul(A, B, C)
        torch.cuda.synchronize()
        name = sg.sg_last_kernel_name()
        if name != "ffma_kernel":
            pytest.skip(f"{name} takes this layout")
        # a multiply-add rounds by 2^-24 of the sum so far: K / 4 of them, three additions
        assert assert_within_bound(C, want, S, "overwrite") <= (K / 4 + 4) * 2.0 ** -24
        sg.sg_matmul(A, B, C, sg.SG_ACCUMULATE)
        assert_within_bound(C, 2 * want, 2 * S, "accumulate")
    assert torch.isnan(wide[:, ::2]).all()
    bias, bv = operand((N,), SEED, 3, "uniform", "f32")
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_matmul_bias_act(A, B, bias, C, sg.SG_ACT_RELU)
    assert_within_bound(C, np.maximum(want + bv, 0), S + np.abs(bv), "bias and relu")
    sg.sg_check()


# Two and three fetches of 128 k, the last by 32 and 64 threads along k.  One chain of additions along k would give another sum: every k but the first adds 1 to
# 2^24, which a chain loses each time, while the three of the four groups that do not hold 2^24 count theirs.
@pytest.mark.parametrize("orders", [("n", "n"), ("t", "t"), ("gaps", "n"), ("t", "gaps")])
@pytest.mark.parametrize("M,N,K", [(5, 33, 257), (33, 31, 287), (1, 7, 299), (7, 5, 129)])
def test_four_short_sums_over_several_fetches(M, N, K, orders):
    A, B = torch.ones(M, K, device="cuda"), torch.ones(K, N, device="cuda")
    A[:, 0] = 2.0 ** 24
    A, B = strided(A, orders[0]), strided(B, orders[1])
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_matmul(A, B, C)
    torch.cuda.synchronize()
    assert sg.sg_last_kernel_name() == "ffma_kernel"
    groups = [len(range(i, K, 4)) for i in range(4)]
    f = np.float32
    want = (f(2 ** 24) + f(groups[1])) + (f(groups[2]) + f(groups[3]))
    assert want > 2 ** 24 + K / 2 and (C == float(want)).all()
    sg.sg_check()


@pytest.mark.parametrize("orders", [("n", "n"), ("t", "t"), ("gaps", "n"), ("t", "gaps")])
@pytest.mark.parametrize("M,N,K", [(5, 33, 257), (33, 31, 287), (1, 7, 299)])
def test_products_of_several_fetches(M, N, K, orders):
    A, a = operand((M, K), SEED, 6, "uniform", "f32")
    B, b = operand((K, N), SEED, 7, "uniform", "f32")
    A, B = strided(A, orders[0]), strided(B, orders[1])
    want, S = ref.matmul(a, b)
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_matmul(A, B, C)
    assert sg.sg_last_kernel_name() == "ffma_kernel"
    assert assert_within_bound(C, want, S, "overwrite") <= (K / 4 + 4) * 2.0 ** -24
    sg.sg_matmul(A, B, C, sg.SG_ACCUMULATE)
    assert_within_bound(C, 2 * want, 2 * S, "accumulate")
    sg.sg_check()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("N,H,W,C,F,KH,KW,s,d", [(1, 29, 29, 3, 64, 3, 3, 2, 1), (1, 7, 5, 5, 33, 5, 3, 1, 1), (2, 9, 11, 3, 32, 3, 3, 1, 2), (3, 1, 2, 1, 1, 1, 1, 1, 1), (1, 6, 6, 9, 31, 5, 5, 1, 1)])
def test_convolutions(N, H, W, C, F, KH, KW, s, d, dtype):
    I, i = operand((N, (H - 1) * s + (KH - 1) * d + 1, (W - 1) * s + (KW - 1) * d + 1, C), SEED, 4, "normal", dtype)
    K, k = operand((KH, KW, C, F), SEED, 5, "normal", dtype)
    want, S = ref.conv2d_nhwc_hwcf(i, k, stride=(s, s), dilation=(d, d))
    O = torch.full((N, H, W + 1, F), float("nan"), device="cuda")[:, :, :W]
    sg.sg_conv2d_nhwc_hwcf(I, K, O, (s, s), (d, d))
    torch.cuda.synchronize()
    assert sg.sg_last_kernel_name() == "ffma_kernel"
    assert assert_within_bound(O, want, S, "conv2d") <= (KH * KW * C / 4 + 4) * 2.0 ** -24
    sg.sg_check()


def test_calls_that_depend_on_each_other():
    """Launches overlap the one ahead: each reads what that one wrote and overwrites what it read."""
    a, b = torch.eye(33, device="cuda")[:, :31].contiguous(), torch.zeros(33, 31, device="cuda")
    eye = torch.eye(31, device="cuda") * 2
    for _ in range(60):
        sg.sg_matmul(a, eye, b)
        assert sg.sg_last_kernel_name() == "ffma_kernel"
        sg.sg_matmul(b, eye * 0.25, a)
    assert torch.equal(a, torch.eye(33, device="cuda")[:, :31])


def test_values_that_are_not_finite():
    A, B = torch.ones(35, 33, device="cuda"), torch.full((33, 37), 0.5, device="cuda")
    A[3, 5], A[4, 6], A[7, 8], A[9, 1], B[2, 4] = float("inf"), float("-inf"), float("nan"), 3.4e38, 2.0
    C = torch.empty(35, 37, device="cuda")
    sg.sg_matmul(A, B, C)
    assert sg.sg_last_kernel_name() == "ffma_kernel"
    want = A.double() @ B.double()
    fine = torch.isfinite(want)
    assert torch.equal(torch.isnan(C), torch.isnan(want)) and torch.equal(torch.isinf(C), torch.isinf(want))
    assert torch.allclose(C[fine].double(), want[fine], rtol=1e-6)


# a grid has up to 65535 tiles along the columns: 32 x 32 tiles end at 2097120 of them, 128 x 128 tiles at 8388480
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("M,N,K", [(1, 2097121, 1), (2, 2097129, 9), (1, 8388479, 1), (1, 8388481, 1), (3, 8388481, 5)])
def test_columns_at_the_limits_of_a_grid(M, N, K, dtype):
    g = torch.Generator(device="cuda").manual_seed(SEED)
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    A, B = (torch.randint(-4, 5, shape, generator=g, device="cuda").to(t) for shape in ((M, K), (K, N)))
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_matmul(A, B, C)
    assert torch.equal(C, (A.double() @ B.double()).float())
    sg.sg_check()
