"""The write-back of a thread block's last tile against the oracle: every tile width, edges that end inside a chunk of 32 columns and
inside a tile of 128 rows, one tile and several per thread block (64-row problems to more tiles than SMs)."""
import pytest
import torch

from helpers import assert_within_bound, operand
from oracle import ref
from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu
SEED = 9500


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("bn,cg", [(64, 1), (128, 1), (256, 1), (128, 2), (256, 2)])
@pytest.mark.parametrize("M,N,K", [(64, 72, 64), (136, 264, 192), (300, 488, 64), (2568, 2056, 64)])
def test_last_tile(M, N, K, bn, cg, dtype):
    if dtype == "f32" and (bn, cg) == (256, 1):
        pytest.skip("no f32 variant of this tile")
    A, a = operand((M, K), SEED, 1, "uniform", dtype)
    B, b = operand((K, N), SEED, 2, "uniform", dtype)
    bias, bias_h = operand((N,), SEED, 3, "normal", "f32")
    wide = torch.full((M, N + 4), float("nan"), device="cuda")
    C = wide[:, :N]
    sg.sg_set_tile_override(bn, cg, 1)
    try:
        sg.sg_matmul(A, B, C)
        torch.cuda.synchronize()
        want, S = ref.matmul(a, b)
        assert_within_bound(C, want, S, "last tile")
        sg.sg_matmul(A, B, C, sg.SG_ACCUMULATE)
        torch.cuda.synchronize()
        assert_within_bound(C, 2 * want, 2 * S, "last tile, accumulate")
        sg.sg_matmul_bias_act(A, B, bias, C, sg.SG_ACT_RELU)
        torch.cuda.synchronize()
        want, S = ref.matmul_bias_act(a, b, bias_h, "relu")
        assert_within_bound(C, want, S, "last tile, bias + relu")
        assert torch.isnan(wide[:, N:]).all()
    finally:
        sg.sg_set_tile_override(0, 0, 0)
    sg.sg_check()
