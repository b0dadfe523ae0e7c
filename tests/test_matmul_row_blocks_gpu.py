"""Row blocks of one fused result multiplied as one product: blocks off a multiple of 8 rows (which a transposed X
would need repacked for), of one row and of none, tiles that span several, cuts over several clusters, exchanged
operands.  Oracle and tolerance as for the other bf16 products (2e-2 relative, 1e-3 absolute against fp64)."""
import pytest
import torch

import paper_2110_15032_b200 as sbp
from test_ops_gpu import _matmul_case

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16
S0, S1 = sbp.S(0), sbp.S(1)


@pytest.mark.parametrize("form", [sbp.SBP_TC_FORM_SPLIT, sbp.SBP_TC_FORM_AUTO])
@pytest.mark.parametrize("M,K,N,k", [(136, 1700, 520, 4), (8, 640, 264, 8), (24, 200, 72, 16), (600, 3001, 136, 8), (1032, 520, 1000, 3)])
def test_row_blocks_of_a_transposed_operand(form, M, K, N, k):
    sbp.sbp_matmul_set_form(form, 0)
    try:
        _matmul_case(M, K, N, k, BF16, S1, S0, ys=S0, tx=True, out_dtype=F32 if N == 264 else BF16)
        _matmul_case(M, K, N, k, BF16, S1, S0, ys=S0, tx=True, flags=sbp.SBP_EPILOGUE_GELU)
        _matmul_case(M, K, N, k, BF16, S1, S0, ys=S0)
    finally:
        sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_AUTO, 0)


def test_row_blocks_cut_over_many_clusters():
    M, K, N, k = 100, 80008, 72, 3
    torch.manual_seed(5)
    X, W = torch.randn(K, M, device="cuda").to(BF16), (torch.randn(K, N, device="cuda") / K ** 0.5).to(BF16)
    xl, wl = ([t.contiguous() for t in torch.tensor_split(T, k, 0)] for T in (X, W))
    for pad in (0, 4):                  # 100 rows are 34 + 33 + 33; X padded to a pitch of 104
        Xp = [torch.nn.functional.pad(t, (0, 4)) for t in xl]
        x = sbp.SbpTensor((K, M), BF16, S0, [t[:, :M] for t in Xp])
        w, y = sbp.SbpTensor((K, N), BF16, S0, wl), sbp.empty_global((M, N), BF16, S0, k)
        room = torch.empty(sbp.sbp_matmul_workspace_bytes(x, w, y, sbp.SBP_TRANS_X) + pad * 10 * M * N * 4, dtype=torch.uint8, device="cuda")
        sbp.sbp_matmul(x, w, y, sbp.SBP_TRANS_X, room if room.numel() else None)
        got, ref = torch.cat([t.double() for t in y.locals]), X.double().T @ W.double()
        assert bool(((got - ref).abs() <= 1e-3 + 2e-2 * ref.abs()).all())
