"""Boxing of unaligned data on either side of the lines at which it takes the shifted 16-byte path, and with one vector a
thread (several destinations) or four: segments of 31 to 33 and 47 to 49 elements and of few aligned pairs, tensors just below and above the element
counts, destinations that are one buffer or many.  Bit-exact against the oracle."""
import pytest
import torch
from test_boxing_disjoint_gpu import _run as run_disjoint
from test_boxing_gpu import _run

import paper_2110_15032_b200 as sbp

pytestmark = pytest.mark.gpu
F32, BF16, I64 = torch.float32, torch.bfloat16, torch.int64
S0, S1, B, P = sbp.S(0), sbp.S(1), sbp.B, sbp.P_SUM


@pytest.mark.parametrize("cols", [91, 94, 97])
@pytest.mark.parametrize("dtype", [F32, BF16, I64])
def test_short_segments(cols, dtype):
    for src, dst in [(S0, S1), (S1, S0), (S1, B), (B, S1)]:
        _run((4801, cols), dtype, src, dst, 3)


@pytest.mark.parametrize("cols", [231, 236, 241])
@pytest.mark.parametrize("dtype", [F32, BF16])
def test_short_segments_of_many_sources(cols, dtype):
    _run((1901, cols), dtype, P, S1, 5)
    _run((1201, cols * 8 // 5), dtype, P, S1, 8)
    run_disjoint((1901, cols), dtype, P, S1, 6, 5)


@pytest.mark.parametrize("units", [31, 33, 55, 57, 63, 65, 119, 121, 129])
@pytest.mark.parametrize("dtype", [F32, BF16])
def test_rows_of_few_pairs(units, dtype):
    for k in (2, 3, 7, 8):
        rows = 1300000 // (2 * units * k) + 1
        _run((rows, 2 * units * k), dtype, P, S1, k)
        _run((rows, 2 * units * k), dtype, S0, S1, k)


@pytest.mark.parametrize("shape", [(631, 633), (635, 637), (893, 895), (895, 899), (1093, 1095), (1097, 1099)])
@pytest.mark.parametrize("dtype", [F32, BF16])
def test_element_counts(shape, dtype):
    for k in (5, 8):
        _run(shape, dtype, P, B, k)
        _run(shape, dtype, P, S0, k)
    run_disjoint(shape, dtype, P, B, 5, 9)
    _run(shape, dtype, S0, B, 5)


@pytest.mark.parametrize("k,q", [(2, 2), (3, 5), (5, 3)])
@pytest.mark.parametrize("shape", [(1021, 401), (3, 500009)])
def test_gathered_integers(shape, k, q):
    _run(shape, I64, S0, B, k)
    _run(shape, I64, S1, B, k)
    run_disjoint(shape, I64, S0, B, k, q)
