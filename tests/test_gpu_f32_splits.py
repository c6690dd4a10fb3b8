"""f32 products on the tensor cores: the converter groups of the narrow tiles against the oracle, and infinities, NaNs and values next to
overflow against f64."""
import numpy as np
import pytest
import torch

from helpers import assert_within_bound, operand
from oracle import ref
from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu
SEED = 9700


# fewer k-blocks than groups, as many, one more, several rounds with a remainder; one tile and more tiles than SMs
@pytest.mark.parametrize("bn,cg,a_t,b_t", [(64, 1, False, False), (64, 1, True, False), (64, 1, False, True), (64, 1, True, True), (128, 2, False, False)])
@pytest.mark.parametrize("M,N,K", [(160, 72, 32), (160, 136, 96), (320, 72, 128), (160, 136, 160), (288, 200, 1056), (4736, 328, 96)])
def test_converter_groups(M, N, K, bn, cg, a_t, b_t):
    A, a = operand((K, M) if a_t else (M, K), SEED, 1, "uniform", "f32")
    B, b = operand((N, K) if b_t else (K, N), SEED, 2, "uniform", "f32")
    A, a = (A.t(), np.ascontiguousarray(a.T)) if a_t else (A, a)
    B, b = (B.t(), np.ascontiguousarray(b.T)) if b_t else (B, b)
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_set_tile_override(bn, cg, 1)
    try:
        sg.sg_matmul(A, B, C)
        torch.cuda.synchronize()
        assert sg.sg_last_kernel_name() == "tc_gemm_kernel<f32>" and tuple(sg.sg_last_tile_choice()) == (bn, cg, 1)
    finally:
        sg.sg_set_tile_override(0, 0, 0)
    want, S = ref.matmul(a, b)
    assert assert_within_bound(C, want, S, "converter groups") < 4e-6      # 2^-19 for the rounded corrections, and the truncating sum
    sg.sg_check()


# an infinity's products are infinities of the right sign (NaN against a zero), a NaN's NaN, and finite values stay finite
@pytest.mark.parametrize("a_t,b_t", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("M,N,K", [(256, 256, 2048), (128, 128, 128)])
def test_special_values(M, N, K, a_t, b_t):
    g = torch.Generator(device="cuda").manual_seed(SEED)
    A = torch.rand(M, K, generator=g, device="cuda") * 2 - 1
    B = torch.rand(K, N, generator=g, device="cuda") * 2 - 1
    A[3, 5], A[4, 6], A[7, 8], A[20, 11] = float("inf"), float("-inf"), float("nan"), 0.0
    A[9, 9], A[10, 9] = torch.finfo(torch.float32).max, -torch.finfo(torch.float32).max
    B[9, :] *= 0.25
    B[5, 7], B[11, 13] = 0.0, float("inf")
    want = A.double() @ B.double()
    a, b = A.t().contiguous().t() if a_t else A, B.t().contiguous().t() if b_t else B
    C = torch.zeros(M, N, device="cuda")
    sg.sg_matmul(a, b, C)
    torch.cuda.synchronize()
    assert torch.equal(torch.isnan(C), torch.isnan(want)) and torch.equal(torch.isinf(C), torch.isinf(want))
    assert torch.equal(torch.sign(C[torch.isinf(C)]), torch.sign(want[torch.isinf(want)]).float())
    bound = A.double().abs().nan_to_num(0, 0, 0) @ B.double().abs().nan_to_num(0, 0, 0)
    finite = torch.isfinite(want)
    assert ((C.double() - want).abs()[finite] <= 4e-6 * bound[finite]).all()
    sg.sg_check()


# An infinity is (largest, infinity) here: its products are infinities of the right sign while its factors are normal and stay below 2000 together
@pytest.mark.parametrize("bn,cg", [(64, 1), (128, 1), (256, 2)])
@pytest.mark.parametrize("a_t,b_t", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("swap", [False, True])
def test_infinities(bn, cg, a_t, b_t, swap):
    M, N, K = 512, 512, 96
    g = torch.Generator(device="cuda").manual_seed(SEED)
    A = torch.rand(M, K, generator=g, device="cuda") * 2 - 1
    B = torch.rand(K, N, generator=g, device="cuda") * 2 - 1
    X, Y = (B.t(), A.t()) if swap else (A, B)
    for i, f in enumerate([1999.25, -1999.25, 1025.5, -0.75, 2.0 ** -126, -(2.0 ** -126)]):
        X[i, 40] = f
    Y[40, 5], Y[40, 6] = float("inf"), float("-inf")
    want = (A.double() @ B.double()).float()
    a, b = A.t().contiguous().t() if a_t else A, B.t().contiguous().t() if b_t else B
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_set_tile_override(bn, cg, 1)
    try:
        sg.sg_matmul(a, b, C)
        torch.cuda.synchronize()
        assert sg.sg_last_kernel_name() == "tc_gemm_kernel<f32>"
    finally:
        sg.sg_set_tile_override(0, 0, 0)
    infinite = torch.isinf(want)
    assert int(infinite.sum()) == 2 * (N if swap else M) and torch.equal(C[infinite], want[infinite])
    assert torch.isfinite(C[~infinite]).all()
    sg.sg_check()


# transposed operands from 128 values of k on: there the correction products are bf16 ones
@pytest.mark.parametrize("bn,cg", [(64, 1), (128, 1), (128, 2), (256, 2)])
@pytest.mark.parametrize("a_t,b_t", [(True, False), (False, True), (True, True)])
@pytest.mark.parametrize("swap", [False, True])
def test_infinities_and_bf16_corrections(bn, cg, a_t, b_t, swap):
    M, N, K = 512, 512, 128
    g = torch.Generator(device="cuda").manual_seed(SEED)
    A = torch.rand(M, K, generator=g, device="cuda") * 2 - 1
    B = torch.rand(K, N, generator=g, device="cuda") * 2 - 1
    X, Y = (B.t(), A.t()) if swap else (A, B)
    for i, f in enumerate([1999.25, -1999.25, 1025.5, -0.75, 2.0 ** -126, -(2.0 ** -126)]):
        X[i, 40] = f
    Y[40, 5], Y[40, 6] = float("inf"), float("-inf")
    want = (A.double() @ B.double()).float()
    a, b = A.t().contiguous().t() if a_t else A, B.t().contiguous().t() if b_t else B
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_set_tile_override(bn, cg, 1)
    try:
        sg.sg_matmul(a, b, C)
        torch.cuda.synchronize()
        assert sg.sg_last_kernel_name() == "tc_gemm_kernel<f32>" and tuple(sg.sg_last_tile_choice()) == (bn, cg, 1)
    finally:
        sg.sg_set_tile_override(0, 0, 0)
    infinite = torch.isinf(want)
    assert int(infinite.sum()) == 2 * (N if swap else M) and torch.equal(C[infinite], want[infinite])
    assert torch.isfinite(C[~infinite]).all()
    sg.sg_check()


@pytest.mark.parametrize("kernel", ["CONV_STRIP", "CONV_WIDE"])
def test_infinities_of_convolutions(kernel):
    I = torch.zeros(2, 40, 41, 16, device="cuda")
    K = torch.full((1, 3, 16, 96), 0.5, device="cuda")
    I[0, 5, 6, 3], I[1, 7, 8, 4], I[1, 20, 21, 2] = float("inf"), float("-inf"), 3.0
    K[0, 1, 3], K[0, 1, 4] = -1999.25, 2.0 ** -126
    O = torch.full((2, 40, 39, 96), float("nan"), device="cuda")
    sg.sg_set_kernel_override(getattr(sg, "SG_KERNEL_" + kernel))
    try:
        sg.sg_conv2d_nhwc_hwcf(I, K, O)
        torch.cuda.synchronize()
        assert sg.sg_last_kernel_name() == f"{kernel.lower()}_kernel<f32>"
    finally:
        sg.sg_set_kernel_override(0)
    want = torch.nn.functional.conv2d(I.double().permute(0, 3, 1, 2), K.double().permute(3, 2, 0, 1)).permute(0, 2, 3, 1).float()
    infinite = torch.isinf(want)
    assert int(infinite.sum()) == 2 * 3 * 96 and torch.equal(O[infinite], want[infinite])
    assert torch.allclose(O[~infinite], want[~infinite], rtol=1e-6, atol=0)
    sg.sg_check()


# transposed operands whose last wave is partly filled: their own k-blocks' price decides on the stream-K tail
@pytest.mark.parametrize("M,N,K,a_t,b_t,accumulate", [(1792, 1664, 1472, False, True, False), (1856, 1792, 2048, True, False, False), (1952, 1184, 1248, True, True, True)])
def test_tail_of_transposed_operands(M, N, K, a_t, b_t, accumulate):
    g = torch.Generator(device="cuda").manual_seed(SEED)
    A = torch.rand((K, M) if a_t else (M, K), generator=g, device="cuda") * 2 - 1
    B = torch.rand((N, K) if b_t else (K, N), generator=g, device="cuda") * 2 - 1
    A, B = A.t() if a_t else A, B.t() if b_t else B
    C = torch.full((M, N), 1.0 if accumulate else float("nan"), device="cuda")
    sg.sg_matmul(A, B, C, sg.SG_ACCUMULATE if accumulate else sg.SG_OVERWRITE)
    torch.cuda.synchronize()
    assert sg.sg_last_stream_k()[1] > 0, "these shapes were meant to take the stream-K tail"
    start = 1.0 if accumulate else 0.0
    err = (C.double() - start - A.double() @ B.double()).abs()
    assert (err <= 4e-6 * (A.double().abs() @ B.double().abs() + start)).all()
    sg.sg_check()
