"""Boxing of data that is not 16-byte aligned, at sizes that take the shifted 16-byte path: rows whose length
leaves every remainder modulo 16 bytes, segments of a few vectors and of many, source and destination buffers
at odd offsets, windows, more sources than are read at once.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch
from helpers import bits, np_bits, osig, split_cpu, to_np
from test_boxing_disjoint_gpu import _run as run_disjoint
from test_boxing_gpu import _run
from test_strided_views_gpu import _outside_untouched, _windows

import paper_2110_15032_b200 as sbp
import sbp_datagen as dg
from oracle import sbp_oracle as O

pytestmark = pytest.mark.gpu

F32, BF16, I64 = torch.float32, torch.bfloat16, torch.int64
S0, S1, B, P, PM = sbp.S(0), sbp.S(1), sbp.B, sbp.P_SUM, sbp.P_MAX
PAIRS = [(S0, S1), (S1, S0), (S0, B), (S1, B), (B, S0), (B, S1), (P, B), (P, S0), (P, S1), (PM, S1), (S0, S0)]


@pytest.mark.parametrize("src,dst", PAIRS)
@pytest.mark.parametrize("dtype", [F32, BF16])
@pytest.mark.parametrize("k", [2, 3, 4, 5, 8])
def test_odd_rows(src, dst, dtype, k):
    _run((1021, 401), dtype, src, dst, k)
    _run((7, 60003 + k), dtype, src, dst, k)
    _run((1009, 403), dtype, src, dst, k, offset_elems=1)      # sources one element off, destinations aligned


@pytest.mark.parametrize("src,dst", [(S0, S1), (S1, S0), (B, S1), (S0, B)])
def test_int64(src, dst):
    _run((1201, 351), I64, src, dst, 3)


@pytest.mark.parametrize("shape", [(61, 67, 103), (9, 11, 65, 67)])
def test_nd(shape):
    for i in range(len(shape)):
        _run(shape, BF16, P, sbp.S(i), 3)
        for j in range(len(shape)):
            if i != j:
                _run(shape, F32, sbp.S(i), sbp.S(j), 3)


@pytest.mark.parametrize("src,dst", [(S0, S0), (S1, S1), (S0, S1), (S1, S0), (S1, B), (P, B), (P, S0), (P, S1), (P, P), (S1, P)])
@pytest.mark.parametrize("p,q", [(3, 2), (2, 5), (7, 3)])
def test_other_placement(src, dst, p, q):
    run_disjoint((1021, 401), F32, src, dst, p, q)
    run_disjoint((643, 647), BF16, src, dst, p, q)


@pytest.mark.parametrize("src_sig,dst_sig", [(S0, S1), (S1, S0), (B, S1), (P, S1), (P, B), (S1, B)])
@pytest.mark.parametrize("dtype", [F32, BF16])
def test_windows(src_sig, dst_sig, dtype):
    shape, k, pad = (701, 601), 3, 7
    src_cpu = [dg.normal(21, r, shape, 0.0, 1.0, dtype) for r in range(k)] if src_sig == P else \
        split_cpu(dg.normal(21, 0, shape, 0.0, 1.0, dtype), src_sig, k)
    want = O.boxing([to_np(t) for t in src_cpu], osig(src_sig), osig(dst_sig), "bf16" if dtype == BF16 else "f32")
    src, _ = _windows(shape, dtype, src_sig, k, pad, fill=src_cpu)
    dst, bufs = _windows(shape, dtype, dst_sig, k, pad)
    sbp.sbp_boxing(src, dst)
    for r in range(k):
        assert np.array_equal(bits(dst.locals[r]), np_bits(want[r], dtype)), f"shard {r} differs"
    _outside_untouched(dst, bufs, pad)
