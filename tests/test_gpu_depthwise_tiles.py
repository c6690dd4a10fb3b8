"""The tiled depthwise kernel at 5 x 5 and 3 x 3 windows, stride 1 and 2: ragged tiles, stacked images, channel blocks of 32 and 64
with remainders, accumulation, a channel slice."""
import numpy as np
import pytest
import torch

from helpers import assert_within_bound, operand
from oracle import ref
from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu
SEED = 9900


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("K,st", [(5, 1), (5, 2), (3, 1), (3, 2)])
@pytest.mark.parametrize("N,Ho,Wo,C", [(1, 1, 1, 16), (40, 7, 7, 200), (70, 5, 6, 96), (3, 33, 17, 72), (2, 65, 40, 24), (9, 14, 31, 128)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_tiles(N, Ho, Wo, C, K, st, dtype, accumulate):
    h_in, w_in = (Ho - 1) * st + K + 1, (Wo - 1) * st + K
    I, i = operand((N, h_in, w_in, C + 8), SEED, 1, "normal", dtype)
    F, f = operand((K, K, C), SEED, 2, "normal", dtype)
    wide = torch.full((N, Ho, Wo, C + 4), float("nan"), device="cuda")
    O = wide[..., :C]
    if accumulate:
        O.fill_(1.0)
    sg.sg_depthwise_conv2d_nhwc_hwc(I[..., 8:], F, O, (st, st), (1, 1), sg.SG_ACCUMULATE if accumulate else sg.SG_OVERWRITE)
    torch.cuda.synchronize()
    if K == 5:
        assert sg.sg_last_kernel_name() == "depthwise_tma_kernel"
    want, S = ref.depthwise_conv2d_nhwc_hwc(np.ascontiguousarray(i[..., 8:]), f, (st, st), (1, 1), out_hw=(Ho, Wo))
    assert_within_bound(O, want + accumulate, S + accumulate, "depthwise tiles")
    assert torch.isnan(wide[..., C:]).all()
    sg.sg_check()
