"""Small fp32 products on the kernel that the library picks for them, the small one or the tiled one: edges of the small kernel's
32 x 32 tile, contractions around one slice a warp, chained segments of uneven length, both stored forms, rows off the 16-byte
rule, replicas.  Oracle and bound as for the other fp32 products.  test_matmul_f32_forms_gpu.py forces each kernel."""
import pytest
import torch

import paper_2110_15032_b200 as sbp
from test_ops_gpu import _matmul_case

pytestmark = pytest.mark.gpu
F32 = torch.float32
S0, S1, B = sbp.S(0), sbp.S(1), sbp.B


@pytest.mark.parametrize("K", [1, 15, 16, 17, 127, 128, 129, 260])
@pytest.mark.parametrize("M,N", [(1, 1), (32, 32), (33, 65), (100, 36), (31, 200)])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, False), (False, True), (True, True)])
def test_tiles_and_slices(M, K, N, tx, tw):
    _matmul_case(M, K, N, 1, F32, B, B, tx=tx, tw=tw)


@pytest.mark.parametrize("M,K,N,k", [(64, 128, 96, 2), (70, 45, 83, 3), (9, 130, 50, 8), (128, 100, 60, 4)])
@pytest.mark.parametrize("ys", [B, S0, S1])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, True)])
def test_groups_and_segments(M, K, N, k, ys, tx, tw):
    _matmul_case(M, K, N, k, F32, S0, B, tx=tx, tw=tw)
    _matmul_case(M, K, N, k, F32, B, S1, tx=tx, tw=tw)
    _matmul_case(M, K, N, k, F32, S1, S0, ys=ys, tx=tx, tw=tw, flags=sbp.SBP_EPILOGUE_GELU if ys == S0 else 0)
