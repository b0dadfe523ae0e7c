"""Results whose rows start anywhere modulo 16 bytes, stored in shifted vectors by both forms of the tensor-core
MatMul: rows shorter than a vector and than a tile's slab, odd pitches, several replicas, row blocks; elements outside
the result stay as they are.  Oracle and tolerance as for the other bf16 products (2e-2 relative, 1e-3 absolute)."""
import pytest
import torch

import paper_2110_15032_b200 as sbp
from test_ops_gpu import _matmul_case

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16
S0, S1, B = sbp.S(0), sbp.S(1), sbp.B


@pytest.fixture(params=[sbp.SBP_TC_FORM_SQUARE, sbp.SBP_TC_FORM_SPLIT])
def form(request):
    sbp.sbp_matmul_set_form(request.param, 0)
    yield
    sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_AUTO, 0)


@pytest.mark.parametrize("N", [1, 7, 9, 63, 65, 127, 130, 300, 513])
@pytest.mark.parametrize("out_dtype", [BF16, F32])
def test_rows_of_any_start(form, N, out_dtype):
    _matmul_case(37, 200, N, 1, BF16, B, B, out_dtype=out_dtype)
    _matmul_case(300, 136, N, 2, BF16, B, B, tw=True, out_dtype=out_dtype, flags=sbp.SBP_EPILOGUE_GELU)
    if N > 8:
        _matmul_case(100, 136, N, 3, BF16, S1, S0, ys=S0, out_dtype=out_dtype)
        _matmul_case(100, 136, N, 3, BF16, S1, S0, ys=S1, out_dtype=out_dtype)
