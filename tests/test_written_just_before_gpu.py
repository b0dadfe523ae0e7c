"""Ids, labels and fp32 operands that one library call writes and the next one reads, with no synchronisation in between: sbp_boxing moves
them into one buffer again and again while lookups, table gradients, losses and products follow on the same stream.  Every kernel
may be set up while the one before it still runs, so each has to wait before it reads."""
import numpy as np
import pytest
import torch

import paper_2110_15032_b200 as sbp
from helpers import make_global, split_cpu, to_np
from oracle import sbp_oracle as O
import sbp_datagen as dg

pytestmark = pytest.mark.gpu
F32, I64 = torch.float32, torch.int64
ROUNDS = 24


def _boxed_each_round(values, n, k):
    """One B buffer, and per round the S(0) tensor that is boxed into it."""
    srcs = [make_global(split_cpu(v, sbp.S(0), k), (n,), I64, sbp.S(0)) for v in values]
    return srcs, sbp.empty_global((n,), I64, sbp.B, k, alias_replicas=True)


@pytest.mark.parametrize("n,rows,dim", [(2400, 500, 32), (70000, 20000, 16), (300, 40, 4)])
def test_ids_written_just_before(n, rows, dim):
    k = 4
    values = [torch.from_numpy(np.random.default_rng(100 + i).integers(0, rows, n)) for i in range(ROUNDS)]
    srcs, ids = _boxed_each_round(values, n, k)
    G, T = dg.normal(61, 0, (n, dim), 0.0, 1.0, F32), dg.normal(61, 1, (rows, dim), 0.0, 1.0, F32)
    go = make_global([G] * k, (n, dim), F32, sbp.B)
    table = make_global(split_cpu(T, sbp.S(0), k), (rows, dim), F32, sbp.S(0))
    outs = [sbp.empty_global((n, dim), F32, sbp.B, k, alias_replicas=True) for _ in range(ROUNDS)]
    grads = [sbp.empty_global((rows, dim), F32, sbp.S(0), k) for _ in range(ROUNDS)]
    torch.cuda.synchronize()
    for i in range(ROUNDS):
        sbp.sbp_boxing(srcs[i], ids)
        sbp.sbp_embedding_backward(go, ids, grads[i])
        sbp.sbp_boxing(srcs[-1 - i], ids)
        sbp.sbp_embedding(table, ids, outs[i])
    torch.cuda.synchronize()
    for i in range(ROUNDS):
        v = values[i].numpy()
        want, mag = O.embedding_grad_table(G.numpy(), v, rows), O.embedding_grad_table(np.abs(G.numpy()), v, rows)
        count = np.bincount(v, minlength=rows)[:, None]
        got = O.from_locals([to_np(t).astype(np.float64) for t in grads[i].locals], O.S0)
        assert np.all(np.abs(got - want) <= count * 2.0 ** -24 * mag + 1e-30), f"round {i}: gradient of other ids"
        assert np.array_equal(to_np(outs[i].locals[0]), T.numpy()[values[-1 - i].numpy()]), f"round {i}: rows of other ids"


@pytest.mark.parametrize("rows,classes", [(64, 4001), (900, 500)])
def test_labels_written_just_before(rows, classes):
    k = 4
    values = [torch.from_numpy(np.random.default_rng(200 + i).integers(0, classes, rows)) for i in range(ROUNDS)]
    srcs, labels = _boxed_each_round(values, rows, k)
    Z = dg.normal(62, 0, (rows, classes), 0.0, 2.0, F32)
    z = make_global(split_cpu(Z, sbp.S(1), k), (rows, classes), F32, sbp.S(1))
    ws = torch.empty(sbp.sbp_softmax_xent_workspace_bytes(z), dtype=torch.uint8, device="cuda")
    vec = lambda: sbp.empty_global((rows,), F32, sbp.B, k, alias_replicas=True)
    losses, m, s = [vec() for _ in range(ROUNDS)], vec(), vec()
    grads = [sbp.empty_global((rows, classes), F32, sbp.S(1), k) for _ in range(ROUNDS)]
    torch.cuda.synchronize()
    for i in range(ROUNDS):
        sbp.sbp_boxing(srcs[i], labels)
        sbp.sbp_softmax_xent(z, labels, losses[i], m, s, ws)
        sbp.sbp_boxing(srcs[-1 - i], labels)
        sbp.sbp_softmax_xent_backward(z, labels, m, s, grads[i])
    torch.cuda.synchronize()
    for i in range(ROUNDS):
        want = O.softmax_xent_logical(Z.numpy(), values[i].numpy())[2]
        assert np.allclose(to_np(losses[i].locals[0]), want, rtol=1e-5, atol=1e-5), f"round {i}: loss of other labels"
        grad = O.from_locals([to_np(t) for t in grads[i].locals], O.S1)
        hit = grad[np.arange(rows), values[-1 - i].numpy()]
        assert np.all(hit < 0.0) and int((grad < 0.0).sum()) == rows, f"round {i}: gradient of other labels"


@pytest.mark.parametrize("form", [sbp.SBP_F32_FORM_TILED, sbp.SBP_F32_FORM_SMALL, sbp.SBP_F32_FORM_TENSOR])
@pytest.mark.parametrize("M,K,N", [(64, 128, 96), (64, 129, 95), (33, 17, 40), (200, 520, 300)])
def test_operands_written_just_before(form, M, K, N):
    """Both operands rewritten between two products that read them; each as the same product of tensors that nothing writes."""
    k = 2
    xs = [make_global(split_cpu(dg.normal(63, i, (M, K), 0.0, 1.0, F32), sbp.S(0), k), (M, K), F32, sbp.S(0)) for i in range(ROUNDS)]
    ws = [make_global(split_cpu(dg.normal(64, i, (K, N), 0.0, 1.0, F32), sbp.S(1), k), (K, N), F32, sbp.S(1)) for i in range(ROUNDS)]
    x, w = sbp.empty_global((M, K), F32, sbp.B, k, alias_replicas=True), sbp.empty_global((K, N), F32, sbp.B, k, alias_replicas=True)
    fixed = []
    for i in range(ROUNDS):
        xi, wi = sbp.empty_global((M, K), F32, sbp.B, k, alias_replicas=True), sbp.empty_global((K, N), F32, sbp.B, k, alias_replicas=True)
        sbp.sbp_boxing(xs[i], xi)
        sbp.sbp_boxing(ws[i], wi)
        fixed.append((xi, wi))
    out, want = ([[sbp.empty_global((M, N), F32, sbp.B, k) for _ in range(2 * ROUNDS)] for _ in range(2)])
    torch.cuda.synchronize()
    sbp.sbp_matmul_set_f32_form(form)
    try:
        for i in range(ROUNDS):
            j = (i + 1) % ROUNDS
            sbp.sbp_matmul(*fixed[i], want[2 * i])
            sbp.sbp_matmul(fixed[j][0], fixed[i][1], want[2 * i + 1])
        torch.cuda.synchronize()
        for i in range(ROUNDS):
            sbp.sbp_boxing(ws[i], w)
            sbp.sbp_boxing(xs[i], x)
            sbp.sbp_matmul(x, w, out[2 * i])
            sbp.sbp_boxing(xs[(i + 1) % ROUNDS], x)
            sbp.sbp_matmul(x, w, out[2 * i + 1])
        torch.cuda.synchronize()
    finally:
        sbp.sbp_matmul_set_f32_form(sbp.SBP_F32_FORM_AUTO)
    for i, (a, b) in enumerate(zip(out, want)):
        assert torch.equal(a.locals[0], b.locals[0]), f"product {i}: of other operands"
