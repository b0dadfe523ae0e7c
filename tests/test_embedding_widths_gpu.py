"""The chunked embedding gather and the scatter of its backward at the edges of their work split: rows of one piece,
of no power of two, of exactly a chunk and of more than one; fewer lookups than a chunk, and counts that leave a
remainder in the last chunk and wave; each chunk length of the scatter.  Gather: bit-exact.  Scatter: the rounding of an
n-term fp32 sum, n u sum|terms| (u = 2^-24)."""
import numpy as np
import pytest
import torch
from helpers import bits, check_guards, make_global, np_bits, split_cpu, to_np

import paper_2110_15032_b200 as sbp
import sbp_datagen as dg
from oracle import sbp_oracle as O

pytestmark = pytest.mark.gpu

F32, BF16, I64 = torch.float32, torch.bfloat16, torch.int64


# 2048 16-byte pieces or 4096 narrower ones fill a chunk: dim 8192 fp32 and 4095 fp32 are the longest rows of theirs,
# 8196 and 4097 * 2 bytes the first too long ones
@pytest.mark.parametrize("dtype,dim,n", [(F32, 4, 1), (F32, 4, 257), (F32, 12, 20001), (F32, 100, 5003), (F32, 8192, 7), (F32, 8196, 7),
                                         (F32, 1, 3000), (F32, 4095, 5), (BF16, 4097, 5), (BF16, 36, 40003), (BF16, 7, 999)])
@pytest.mark.parametrize("k,alias", [(1, False), (3, True), (3, False)])
def test_gather_widths(dtype, dim, n, k, alias):
    rows = 203
    table = dg.uniform(1005, 20, (rows, dim), -0.05, 0.05, dtype)
    table[5, dim - 1] = -0.0
    ids = dg.zipf_ids(1005, 21, (n,), rows, 1.05)
    ids[n // 2] = rows
    ids[n - 1] = rows if n == 1 else 5
    tab = make_global(split_cpu(table, sbp.S(0), k), (rows, dim), dtype, sbp.S(0))
    idt = make_global([ids] * k, (n,), I64, sbp.B)
    out = sbp.empty_global((n, dim), dtype, sbp.B, k, alias_replicas=alias)
    for t in out.locals:
        t.view(torch.uint8).fill_(0x5A)
    oob = torch.zeros(1, dtype=torch.int32, device="cuda")
    sbp.sbp_embedding(tab, idt, out, oob)
    torch.cuda.synchronize()
    check_guards()
    want = O.embedding_logical(to_np(table), ids.numpy())
    if k > 1:
        want = want + np.float32(0.0)
    for t in out.locals:
        assert np.array_equal(bits(t), np_bits(want, dtype))
    assert int(oob.item()) == 1


# 113 664 and 227 328 lookups are where chunks of 512 and 1024 begin (rows of 16 and 8 vectors at most)
@pytest.mark.parametrize("dim,n", [(4, 1), (4, 255), (12, 113663), (64, 113664), (68, 113664), (20, 227327), (32, 227328), (36, 227329), (128, 3001)])
@pytest.mark.parametrize("k", [1, 3])
def test_scatter_chunks(dim, n, k):
    rows = 3001
    ids = dg.zipf_ids(1005, 22, (n,), rows, 1.05)
    ids[n - 1] = rows
    G = dg.normal(1005, 23, (n, dim), 0.0, 1.0, F32)
    go = make_global([G] * k, (n, dim), F32, sbp.B)
    idt = make_global([ids] * k, (n,), I64, sbp.B)
    gt = sbp.empty_global((rows, dim), F32, sbp.S(0), k)
    for t in gt.locals:
        t.fill_(float("nan"))
    oob = torch.zeros(1, dtype=torch.int32, device="cuda")
    sbp.sbp_embedding_backward(go, idt, gt, oob)
    torch.cuda.synchronize()
    assert int(oob.item()) == 1
    want = O.embedding_grad_table(G.numpy(), ids.numpy(), rows)
    mag = O.embedding_grad_table(np.abs(G.numpy()), ids.numpy(), rows)
    counts = O.embedding_grad_table(np.ones((n, 1)), ids.numpy(), rows)
    got = O.from_locals([to_np(t).astype(np.float64) for t in gt.locals], O.S0)
    assert np.all(np.abs(got - want) <= counts * 2.0 ** -24 * mag + 1e-30)
    assert np.all(got[counts[:, 0] == 0] == 0.0)
