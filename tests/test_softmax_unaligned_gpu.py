"""Split softmax cross entropy, forward and backward, where rows start at every remainder modulo 16 bytes: class
counts around a vector, a chunk and a span, shards shorter than a vector, few rows (spans cut finer) and many,
windows whose logits and gradient stand alike modulo 16 and not.  Oracle and tolerance as for the other softmax
tests (row max exact; 2e-2 relative, 1e-3 absolute)."""
import numpy as np
import pytest
import torch
from helpers import assert_close, make_global, split_cpu, to_np

import paper_2110_15032_b200 as sbp
import sbp_datagen as dg
from oracle import sbp_oracle as O

pytestmark = pytest.mark.gpu

F32, BF16, I64 = torch.float32, torch.bfloat16, torch.int64


def _case(rows, classes, k, dtype, pad=(0, 0)):
    Z = dg.normal(61, rows, (rows, classes), 0.0, 2.0, dtype)
    labels = dg.integers(62, rows, (rows,), 0, classes)
    labels[:2] = torch.tensor([0, classes - 1])[:rows]          # the elements before and after the whole vectors
    zl = split_cpu(Z, sbp.S(1), k)

    def windows(pad, fill):
        out = []
        for t in zl:
            buf = torch.full((t.shape[0], t.shape[1] + pad), 7.0, dtype=dtype, device="cuda")
            w = buf[:, pad // 2:pad // 2 + t.shape[1]]
            if fill:
                w.copy_(t)
            out.append(w)
        return sbp.SbpTensor((rows, classes), dtype, sbp.S(1), out)

    logits = windows(pad[0], True) if pad[0] else make_global(zl, (rows, classes), dtype, sbp.S(1))
    grad = windows(pad[1], False) if pad[1] else sbp.empty_global((rows, classes), dtype, sbp.S(1), k)
    lab = make_global([labels] * k, (rows,), I64, sbp.B)
    loss, rmax, rsum = [sbp.empty_global((rows,), F32, sbp.B, k) for _ in range(3)]
    ws = torch.empty(max(4, sbp.sbp_softmax_xent_workspace_bytes(logits)), dtype=torch.uint8, device="cuda")
    sbp.sbp_softmax_xent(logits, lab, loss, rmax, rsum, ws)
    sbp.sbp_softmax_xent_backward(logits, lab, rmax, rsum, grad)
    torch.cuda.synchronize()
    locs = O.to_locals(to_np(Z), O.S1, k)
    m, S, ref = O.softmax_xent_split(locs, labels.numpy())
    want = O.to_locals(O.softmax_xent_grad(to_np(Z), labels.numpy()), O.S1, k)
    for r in range(k):
        assert np.array_equal(to_np(rmax.locals[r]), m.astype(np.float32))
        assert_close(to_np(rsum.locals[r]), S, 2e-2, 1e-3, "row sum")
        assert_close(to_np(loss.locals[r]), ref, 2e-2, 1e-3, "loss")
        assert_close(to_np(grad.locals[r]), want[r], 2e-2, 1e-3, "gradient")


@pytest.mark.parametrize("dtype", [F32, BF16])
@pytest.mark.parametrize("classes,k", [(2, 1), (7, 2), (9, 4), (31, 2), (1003, 3), (4097, 1), (16395, 2), (32771, 1), (70001, 4)])
@pytest.mark.parametrize("rows", [1, 5, 70])
def test_class_counts(rows, classes, k, dtype):
    _case(rows, classes, k, dtype)


@pytest.mark.parametrize("dtype", [F32, BF16])
@pytest.mark.parametrize("pad", [(3, 3), (8, 0), (3, 5), (0, 11)])
def test_windows(dtype, pad):
    _case(19, 2003, 2, dtype, pad)


@pytest.mark.parametrize("dtype", [F32, BF16])
def test_few_rows_many_classes(dtype):
    _case(3, 400003, 2, dtype)
    _case(2, 262144, 8, dtype)


@pytest.mark.parametrize("dtype", [F32, BF16])
@pytest.mark.parametrize("rows", [739, 740, 1481, 2961])
def test_many_rows(rows, dtype):
    _case(rows, 333, 3, dtype)
    _case(rows, 11, 8, dtype)
