"""The kernel for small problems on infinities and on values next to overflow, in either operand, against factors that a split does not carry
beside infinities: low parts above one half, subnormals.  Both of its f32 forms; every entry against f64 rounded to f32."""
import pytest
import torch

from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu
INF, MAX = float("inf"), torch.finfo(torch.float32).max
FACTORS = [4098.5, -4098.5, 9005.0, -9005.0, 1e30, -1e30, 2.0 ** -140, -(2.0 ** -149), 0.5]


# (the plain layout runs as tf32 and bf16 parts, the others as three bf16 parts; 16-row and 32-row tiles)
@pytest.mark.parametrize("a_t,b_t", [(False, False), (True, False), (False, True)])
@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("M,N,K", [(128, 128, 128), (1600, 96, 72)])
def test_products(M, N, K, a_t, b_t, swap):
    g = torch.Generator(device="cuda").manual_seed(9900)
    A = torch.rand(M, K, generator=g, device="cuda") * 2 - 1
    B = torch.rand(K, N, generator=g, device="cuda") * 2 - 1
    X, Y = (B.t(), A.t()) if swap else (A, B)       # the factors in X's rows, what they meet in Y's columns
    for i, f in enumerate(FACTORS):
        X[i, 3] = f
    Y[3, 5], Y[3, 6] = INF, -INF
    X[40, 9] = MAX
    for j, f in enumerate(FACTORS[:6]):            # (a subnormal's parts are multiples of 2^-136: that shows beside the largest value)
        Y[9, 32 + j] = f
    Y[11, 50], Y[12, 50] = 1e38, -1e38             # finite products of either sign that overflow
    X[50, 11], X[51, 12] = 9005.0, 9005.0
    X[60, 13] = float("nan")
    want = (A.double() @ B.double()).float()
    a, b = A.t().contiguous().t() if a_t else A, B.t().contiguous().t() if b_t else B
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_matmul(a, b, C)
    torch.cuda.synchronize()
    assert sg.sg_last_kernel_name() == "small_gemm_kernel<f32>"
    infinite, nan = torch.isinf(want), torch.isnan(want)
    assert infinite.any() and int(nan.sum()) == (M if swap else N) and torch.equal(torch.isnan(C), nan)
    assert torch.equal(torch.isinf(C), infinite) and torch.equal(C[infinite], want[infinite])
    bound = A.double().abs().nan_to_num(0, 0, 0) @ B.double().abs().nan_to_num(0, 0, 0)
    err = (C.double() - A.double().nan_to_num(0, 0, 0) @ B.double().nan_to_num(0, 0, 0)).abs()
    finite = ~(infinite | nan)
    # two corrections of up to 2^-11 of their product with both factors rounded by 2^-9 (a large factor's product is the whole sum: nothing averages) 2^-18,
    # the dropped product 2^-22, some twenty truncating or rounding additions 2^-24 each
    assert (err[finite] <= (2.0 ** -18 + 2.0 ** -22 + 20 * 2.0 ** -24) * bound[finite]).all()
    sg.sg_check()
