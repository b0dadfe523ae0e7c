"""Two-axis boxing with its groups in one launch: more groups than one launch holds, groups of uneven and zero rows,
groups whose data is not aligned alike (launched apart) and unaligned ones large enough for shifted vectors.  Bit-exact."""
import numpy as np
import pytest
import torch
from helpers import bits, np_bits, osig, to_np
import test_two_axis_gpu as small

import paper_2110_15032_b200 as sbp
import sbp_datagen as dg
from oracle import sbp_oracle as O

pytestmark = pytest.mark.gpu

F32, BF16 = torch.float32, torch.bfloat16
S0, S1, B, P = sbp.S(0), sbp.S(1), sbp.B, sbp.P_SUM


@pytest.mark.parametrize("src_sigs,dst_sigs", small.BOX2)
@pytest.mark.parametrize("pshape", [(5, 3), (8, 2)])
def test_more_groups_than_one_launch_holds(src_sigs, dst_sigs, pshape):
    small.test_two_axis_boxing_one_axis_at_a_time(src_sigs, dst_sigs, pshape, BF16)


@pytest.mark.parametrize("rows,cols", [(2 * 1001 + 1, 607), (1, 65), (3, 8), (2 * 500, 1024)])
@pytest.mark.parametrize("src,dst", [(P, B), (P, S1), (S1, B), (S0, S1)])
@pytest.mark.parametrize("dtype", [F32, BF16])
def test_groups_inside_axis_one(rows, cols, src, dst, dtype):
    k0, k1 = 2, 3
    st = "f32" if dtype == F32 else "bf16"
    src_np, want = [], []
    for i in range(k0):
        gshape = sbp.sbp_local_shape((rows, cols), S0, k0, i, dtype)
        full = [to_np(dg.normal(4100, 10 * i + j, gshape, 0, 1, dtype)) for j in range(k1)]
        parts = full if src == P else O.to_locals(full[0], osig(src), k1)
        src_np += parts
        want += O.boxing(parts, osig(src), osig(dst), st) if gshape[0] > 0 else [None] * k1
    s = sbp.SbpTensor((rows, cols), dtype, (S0, src), [torch.from_numpy(np.ascontiguousarray(a)).to(dtype).cuda() for a in src_np], (k0, k1))
    d = sbp.empty_global((rows, cols), dtype, (S0, dst), (k0, k1))
    for t in d.locals:
        t.view(torch.uint8).fill_(0xAB)
    sbp.sbp_boxing(s, d)
    torch.cuda.synchronize()
    sbp.sbp_check_device_errors()
    for r in range(k0 * k1):
        if want[r] is not None:
            assert np.array_equal(bits(d.locals[r]), np_bits(want[r], dtype)), f"device {r}"
