"""Embedding calls whose shape decides how they are dealt out.  Table gradients of long rows and few lookups, whose columns are
dealt out to several CTAs: one pass of 32 vectors and one vector more, more CTAs than columns, ids outside the table (counted
once, not once a CTA), every chunk's last position; bound of an n-term fp32 sum: n u sum|terms|, u = 2^-24.  Lookups of short
rows, and results just below and above the size at which several replicas are written element by element."""
import numpy as np
import pytest
import torch

import paper_2110_15032_b200 as sbp
import sbp_datagen as dg
from helpers import make_global, to_np
from oracle import sbp_oracle as O

pytestmark = pytest.mark.gpu
F32, I64 = torch.float32, torch.int64


@pytest.mark.parametrize("rows,dim,lookups", [(40, 128, 300), (40, 132, 300), (7, 256, 1), (100, 4000, 257), (2000, 8192, 100), (30, 40000, 64), (500, 1000, 3000)])
@pytest.mark.parametrize("k", [1, 3])
def test_gradient_of_long_rows(rows, dim, lookups, k):
    ids = torch.from_numpy(np.random.default_rng(dim).integers(0, rows, lookups))
    outside = 0
    if lookups > 10:
        ids[3], ids[lookups - 1], outside = -1, rows, 2
    G = dg.normal(71, 0, (lookups, dim), 0.0, 1.0, F32)
    gt = sbp.empty_global((rows, dim), F32, sbp.S(0), k)
    for t in gt.locals:
        t.fill_(float("nan"))
    oob = torch.zeros(1, dtype=torch.int32, device="cuda")
    sbp.sbp_embedding_backward(make_global([G] * k, (lookups, dim), F32, sbp.B), make_global([ids] * k, (lookups,), I64, sbp.B), gt, oob)
    assert int(oob.item()) == outside
    want, mag = O.embedding_grad_table(G.numpy(), ids.numpy(), rows), O.embedding_grad_table(np.abs(G.numpy()), ids.numpy(), rows)
    count = np.bincount(ids[(ids >= 0) & (ids < rows)].numpy(), minlength=rows)[:, None]
    got = O.from_locals([to_np(t).astype(np.float64) for t in gt.locals], O.S0)
    assert np.all(np.abs(got - want) <= count * 2.0 ** -24 * mag + 1e-30)


@pytest.mark.parametrize("dtype", [F32, torch.bfloat16])
@pytest.mark.parametrize("dim", [1, 3, 4, 12])
@pytest.mark.parametrize("lookups", [1, 255, 5000, 150001])
def test_lookup_of_short_rows_to_several_replicas(dtype, dim, lookups):
    """Chunks of 256 lookups whose pieces fill only the first of a thread's steps."""
    rows, k = 4001, 3
    T = dg.normal(72, 0, (rows, dim), 0.0, 1.0, dtype)
    ids = torch.from_numpy(np.random.default_rng(lookups).integers(0, rows, lookups))
    table = sbp.SbpTensor((rows, dim), dtype, sbp.S(0), [t.contiguous().cuda() for t in torch.tensor_split(T, k, 0)])
    out = sbp.empty_global((lookups, dim), dtype, sbp.B, k)
    sbp.sbp_embedding(table, make_global([ids] * k, (lookups,), I64, sbp.B), out)
    for t in out.locals:
        assert torch.equal(t.cpu(), T[ids])


@pytest.mark.parametrize("lookups", [292968, 292969, 300001])
def test_large_results_to_four_replicas(lookups):
    rows, dim, k = 3001, 128, 4
    T = torch.randn(rows, dim, device="cuda")
    ids = torch.randint(0, rows, (lookups,), device="cuda")
    ids[5] = rows
    oob = torch.zeros(1, dtype=torch.int32, device="cuda")
    table = sbp.SbpTensor((rows, dim), F32, sbp.S(0), [t.contiguous() for t in torch.tensor_split(T, k, 0)])
    out = sbp.empty_global((lookups, dim), F32, sbp.B, k)
    sbp.sbp_embedding(table, sbp.SbpTensor((lookups,), I64, sbp.B, [ids] * k), out, oob)
    want = torch.cat([T, torch.zeros(1, dim, device="cuda")])[ids]
    assert int(oob.item()) == 1
    for t in out.locals:
        assert torch.equal(t, want)
