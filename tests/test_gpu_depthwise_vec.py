"""Small 3 x 3 depthwise layers of stride 2 (and any stride and dilation down the rows) and channel blocks of 64 against the oracle: one to a
few output columns per thread, channel counts around a thread's four."""
import pytest

from helpers import assert_within_bound
from paper_2202_03293_b200 import binding as sg
from test_gpu_depthwise import run2d

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("N,Ho,Wo,C,st,dl", [(1, 1, 1, 4, (2, 2), (1, 1)), (2, 3, 2, 12, (2, 2), (1, 1)), (1, 7, 7, 24, (2, 2), (1, 1)), (3, 5, 3, 20, (1, 2), (2, 1)),
                                              (4, 4, 9, 64, (3, 2), (1, 1)), (2, 6, 5, 16, (1, 1), (1, 1)), (1, 13, 31, 100, (2, 2), (1, 1))])
def test_small_layers(N, Ho, Wo, C, st, dl, accumulate, dtype):
    O, want, S = run2d(N, Ho, Wo, C, 3, 3, st, dl, dtype, accumulate, extra=(1, 1))
    assert_within_bound(O, want, S, "depthwise, small")
    sg.sg_check()


# bf16 channel counts on both sides of the line between blocks of 64 and of 32
@pytest.mark.parametrize("C", [72, 96, 104, 136, 160, 200, 416])
@pytest.mark.parametrize("s,K", [(1, 3), (2, 3), (2, 5)])
def test_channel_blocks(C, s, K):
    O, want, S = run2d(6, 21, 27, C, K, K, (s, s), (1, 1), "bf16")
    assert_within_bound(O, want, S, "depthwise, channel blocks")
    sg.sg_check()
