"""Copies of dense tensors, which move as rows of 256 elements, and transposes on both sides of the size from which fewer tiles
are in flight: bit patterns come out unchanged and nothing around the destination is written."""
import pytest
import torch

from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu
FILL = -7


def run(op, R, C, dtype, src_pitch, dst_pitch):
    bits = torch.int16 if dtype == torch.bfloat16 else torch.int32
    n_r, n_c = (C, R) if op == "transpose" else (R, C)
    g = torch.Generator(device="cuda").manual_seed(R * 31 + C)
    src = torch.randint(-30000, 30000, (R, src_pitch), dtype=bits, device="cuda", generator=g)
    dst = torch.full((n_r + 1, dst_pitch), FILL, dtype=bits, device="cuda")
    (sg.sg_transpose2d if op == "transpose" else sg.sg_copy2d)(src.view(dtype)[:, :C], dst.view(dtype)[:n_r, :n_c])
    torch.cuda.synchronize()
    sg.sg_check()
    assert sg.sg_last_kernel() == sg.SG_KERNEL_TMA_MOVE
    want = src[:, :C].t() if op == "transpose" else src[:, :C]
    assert torch.equal(dst[:n_r, :n_c], want)
    assert bool((dst[n_r:] == FILL).all()) and bool((dst[:, n_c:] == FILL).all())


# one row; rows shorter than 256; totals that are and are not multiples of 256; the last box cut off; a pitch on either side
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("R,C,src_pad,dst_pad", [(1, 256, 0, 0), (1, 256 * 37, 0, 0), (1, 264, 0, 0), (32, 24, 0, 0), (33, 24, 0, 0),
                                                 (256 * 9, 8, 0, 0), (250, 1024, 0, 0), (1031, 512, 0, 0), (1031, 512, 8, 0), (1031, 512, 0, 8),
                                                 (3000, 1016, 0, 0), (2, 65536, 0, 0)])
def test_dense_copies(R, C, src_pad, dst_pad, dtype):
    run("copy", R, C, dtype, C + src_pad, C + dst_pad)


# 64 MB in elements of 4 and of 2 bytes, less one row of tiles and exactly; tiles cut off on both sides
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("R,C", [(4096, 4096), (4088, 4104), (8192, 4096), (8184, 4088), (128, 64), (136, 72), (8, 2048)])
def test_transposes_around_the_window_rule(R, C, dtype):
    run("transpose", R, C, dtype, C, R)


# Few tiles: the number of thread blocks that an SM may hold goes by the tiles (148 SMs), on either side of each line: 128 rows by 128 bytes where TMA
# moves them, 32 x 32 where a row does not start on 16 bytes
@pytest.mark.parametrize("dtype,es", [(torch.float32, 4), (torch.bfloat16, 2)])
@pytest.mark.parametrize("tiles", [148, 149, 185, 186, 296, 297, 444, 445, 740, 889, 1184, 1190])
@pytest.mark.parametrize("aligned", [True, False])
def test_transposes_of_few_tiles(tiles, aligned, dtype, es):
    a = max(d for d in range(1, 21) if tiles % d == 0)
    R, C = (128 * a, 128 // es * (tiles // a)) if aligned else (32 * a - 5, 32 * (tiles // a) - 3)
    src = torch.randint(-2 ** 15, 2 ** 15, (R, C * es // 2), device="cuda", dtype=torch.int16).view(dtype)
    dst = torch.zeros(C, R, device="cuda", dtype=dtype)
    for _ in range(3):
        sg.sg_transpose2d(src, dst)
    assert sg.sg_last_kernel_name() == ("transpose_tma_kernel" if aligned else "tile_move_kernel")
    bits = torch.int32 if es == 4 else torch.int16
    assert torch.equal(dst.view(bits), src.view(bits).t())
    sg.sg_check()


# 64 x 64 tiles, on either side of five and six to an SM (148 SMs), where tiles of 4 bytes are loaded another way; the last ones cut off
@pytest.mark.parametrize("dtype,bits", [(torch.float32, torch.int32), (torch.bfloat16, torch.int16)])
@pytest.mark.parametrize("a,b", [(20, 37), (19, 39), (24, 37), (7, 127), (1, 741)])
@pytest.mark.parametrize("cut", [0, 1, 31, 63])
def test_unaligned_transposes_of_five_and_six_tiles_to_an_sm(a, b, cut, dtype, bits):
    R, C = 64 * a - cut, 64 * b - cut
    src = torch.randint(-30000, 30000, (R, C + 1 + C % 2), dtype=bits, device="cuda")       # odd pitches
    dst = torch.full((C + 1, R + 1 + R % 2), FILL, dtype=bits, device="cuda")
    sg.sg_transpose2d(src.view(dtype)[:, :C], dst.view(dtype)[:C, :R])
    assert sg.sg_last_kernel_name() == "tile_move_kernel"
    assert torch.equal(dst[:C, :R], src[:, :C].t())
    assert bool((dst[C:] == FILL).all()) and bool((dst[:, R:] == FILL).all())
    sg.sg_check()
