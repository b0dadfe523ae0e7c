"""Products of at most four K-blocks of 64, and one more: many tiles a CTA pair, so that every staging slab and ring slot
comes round, ragged edges, both epilogues.  Oracle and tolerance as for the other bf16 products (2e-2 relative, 1e-3
absolute against fp64)."""
import pytest
import torch

import paper_2110_15032_b200 as sbp
from test_ops_gpu import _matmul_case

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


@pytest.mark.parametrize("K", [8, 64, 128, 200, 256, 264])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, False), (False, True), (True, True)])
def test_short_contractions(K, tx, tw):
    sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_SQUARE, 3)      # three pairs: six or more tiles each
    try:
        _matmul_case(1000, K, 1304, 1, BF16, sbp.B, sbp.B, tx=tx, tw=tw, flags=sbp.SBP_EPILOGUE_GELU if K == 128 else 0,
                     out_dtype=F32 if K == 200 else BF16)
    finally:
        sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_AUTO, 0)
