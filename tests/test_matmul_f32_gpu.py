"""fp32 products on the kernel that the library picks, where they can go wrong: edges of tiles, K-slices with a
remainder, contractions split over a cluster, chained segments of uneven and zero length, operands that
miss the 16-byte rule, both stored forms of either operand.  Same oracle and the same bound
(probabilistic bound on recursive summation) as the other fp32 products.  test_matmul_f32_forms_gpu.py forces each kernel."""
import pytest
import torch

import paper_2110_15032_b200 as sbp
from test_ops_gpu import _matmul_case

pytestmark = pytest.mark.gpu
F32 = torch.float32
S0, S1, B, P = sbp.S(0), sbp.S(1), sbp.B, sbp.P_SUM


@pytest.mark.parametrize("M,K,N", [(1, 1, 1), (64, 16, 64), (65, 17, 63), (128, 48, 128), (129, 1000, 127), (40, 2500, 24),
                                   (257, 20, 1030), (1150, 200, 1300)])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, True)])
def test_tile_edges_and_split_contractions(M, K, N, tx, tw):
    _matmul_case(M, K, N, 1, F32, B, B, tx=tx, tw=tw)
    _matmul_case(M, K, N, 3, F32, S0, B, tx=tx, tw=tw)


@pytest.mark.parametrize("M,K,N,k", [(70, 1003, 90, 3), (130, 3, 70, 8), (33, 2048, 257, 4)])
@pytest.mark.parametrize("ys", [B, S0, S1])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, False), (False, True)])
def test_chained_segments(M, K, N, k, ys, tx, tw):
    _matmul_case(M, K, N, k, F32, S1, S0, ys=ys, tx=tx, tw=tw, flags=sbp.SBP_EPILOGUE_GELU if ys == S1 else 0)


def test_split_contraction_gives_the_same_bits_every_time():
    X = torch.randn(100, 4000, device="cuda")
    W = torch.randn(4000, 90, device="cuda")
    x, w = sbp.SbpTensor((100, 4000), F32, B, [X]), sbp.SbpTensor((4000, 90), F32, B, [W])
    y = sbp.empty_global((100, 90), F32, B, 1)
    sbp.sbp_matmul(x, w, y)
    ref = y.locals[0].clone()
    for _ in range(20):
        sbp.sbp_matmul(x, w, y)
        assert torch.equal(ref, y.locals[0])
