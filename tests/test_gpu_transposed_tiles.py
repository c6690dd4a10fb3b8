"""Operands stored transposed: every tile that is built for them, and (f32) the reductions on either side of the line from which
the correction products run in bf16."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from helpers import assert_within_bound, operand
from oracle import ref
from paper_2202_03293_b200 import binding as sg

pytestmark = pytest.mark.gpu
SEED = 9750


# a k-block is 32 values (f32) or 64 (bf16): one, the last with three tf32 products, the first with bf16 corrections, a remainder;
# one ragged tile, and more tiles than SMs
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("a_t,b_t", [(True, False), (False, True), (True, True)])
@pytest.mark.parametrize("bn,cg", [(64, 1), (128, 1), (128, 2), (256, 2)])
@pytest.mark.parametrize("M,N,K", [(320, 264, 32), (320, 264, 96), (320, 264, 128), (320, 264, 168), (5120, 1096, 136)])
def test_transposed_tiles(M, N, K, bn, cg, a_t, b_t, dtype):
    A, a = operand((K, M) if a_t else (M, K), SEED, 1, "uniform", dtype)
    B, b = operand((N, K) if b_t else (K, N), SEED, 2, "uniform", dtype)
    A, a = (A.t(), np.ascontiguousarray(a.T)) if a_t else (A, a)
    B, b = (B.t(), np.ascontiguousarray(b.T)) if b_t else (B, b)
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_set_tile_override(bn, cg, 1)
    try:
        sg.sg_matmul(A, B, C)
        torch.cuda.synchronize()
        name, choice = sg.sg_last_kernel_name(), tuple(sg.sg_last_tile_choice())
    finally:
        sg.sg_set_tile_override(0, 0, 0)
    assert name == f"tc_gemm_kernel<{dtype}>"
    if (bn, cg) != (128, 2) or (dtype == "f32" and K >= 128):      # (else not built)
        assert choice == (bn, cg, 1)
    rows = np.unique(np.r_[0:M:max(1, M // 40), M - 1])
    want, S = ref.matmul(np.ascontiguousarray(a[rows]), b)
    assert assert_within_bound(C[torch.from_numpy(rows).cuda()], want, S, "transposed tiles") < 4e-6      # 2^-19 for the rounded corrections, and the truncating sum
    sg.sg_check()


# One product a sum, so that nothing hides its own error: three tf32 products below 128 values of k, bf16 corrections from there on.  A factor is hi + lo,
# lo up to 2^-11 of it; rounding lo to tf32 moves it by 2^-12, to bf16 by 2^-9, hi to bf16 by 2^-8; lo * lo is dropped, up to 2^-22, and three
# truncating additions take up to 2^-23 each (the first adds to zero).
@pytest.mark.parametrize("K", [97, 100, 124, 127, 128, 160])
@pytest.mark.parametrize("a_t,b_t", [(True, False), (False, True), (True, True)])
@pytest.mark.parametrize("bn", [64, 128])
def test_single_products(K, a_t, b_t, bn):
    if (b_t or not a_t) and K % 4:
        pytest.skip("rows of K values do not start on 16-byte boundaries")
    M, N = 512, 512
    g = torch.Generator(device="cuda").manual_seed(K)
    A, B = torch.zeros(M, K, device="cuda"), torch.rand(K, N, generator=g, device="cuda") + 1
    A[torch.arange(M), torch.randint(0, K, (M,), generator=g, device="cuda")] = torch.rand(M, generator=g, device="cuda") + 1
    a, b = A.t().contiguous().t() if a_t else A, B.t().contiguous().t() if b_t else B
    C = torch.full((M, N), float("nan"), device="cuda")
    sg.sg_set_tile_override(bn, 1, 1)
    try:
        sg.sg_matmul(a, b, C)
        torch.cuda.synchronize()
        assert sg.sg_last_kernel_name() == "tc_gemm_kernel<f32>" and tuple(sg.sg_last_tile_choice()) == (bn, 1, 1)
    finally:
        sg.sg_set_tile_override(0, 0, 0)
    want = A.double() @ B.double()
    factor = 2.0 ** -23 if K < 128 else 2.0 ** -20 + 2.0 ** -19
    assert ((C.double() - want).abs() <= (2 * factor + 2.0 ** -22 + 2 * 2.0 ** -23) * want).all()
    sg.sg_check()


_CHOICES = """
import json, sys, torch
from paper_2202_03293_b200 import binding as sg
out = []
for M, N, K, fused in json.loads(sys.argv[1]):
    for a_t, b_t in ((True, False), (False, True), (True, True)):
        A, B = torch.zeros((K, M) if a_t else (M, K), device="cuda"), torch.zeros((N, K) if b_t else (K, N), device="cuda")
        A, B, C = A.t() if a_t else A, B.t() if b_t else B, torch.empty(M, N, device="cuda")
        if fused:
            sg.sg_matmul_bias_act(A, B, torch.zeros(N, device="cuda"), C, sg.SG_ACT_RELU)
        else:
            sg.sg_matmul(A, B, C)
        out.append([sg.sg_last_kernel_name(), sg.sg_last_tile_choice()[2]])
sg.sg_check()
print(json.dumps(out))
"""


def test_ranges_are_as_short_as_their_error_asks():
    """A range of k gets at most half as long again as three tf32 products would have had, also where a consumer takes the sum."""
    shapes = [[512, 512, 384], [512, 512, 416], [512, 1024, 512], [256, 512, 1024], [256, 256, 1024], [512, 512, 2048], [1024, 1024, 512], [256, 256, 4096]]
    shapes = [s + [f] for s in shapes for f in (0, 1)]
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    found = []
    for mix in ("1", "0"):
        r = subprocess.run([sys.executable, "-c", _CHOICES, json.dumps(shapes)], cwd=root, env={**os.environ, "SG_TC_MIX": mix}, capture_output=True,
                           text=True, timeout=300)
        assert r.returncode == 0, r.stderr
        found.append(json.loads(r.stdout))
    for i, ((name, shares), (name0, shares0)) in enumerate(zip(*found)):
        M, N, K, fused = shapes[i // 3]
        assert name == name0 == "tc_gemm_kernel<f32>"
        kb = K // 32
        assert -(-kb // shares) <= -(-kb // shares0) * 3 // 2, (M, N, K, fused, shares, shares0)
