"""The fused classifier at logits of any size: sums and gradients depend on differences from the row's maximum alone.  Both of
its kernels, rows in the tens (few rows) and the hundreds."""
import pytest
import torch

import paper_2110_15032_b200 as sbp

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


@pytest.mark.parametrize("top", [0.0, 2.0 ** 13, -2.0 ** 13, 2.0 ** 20, -2.0 ** 20, 2.0 ** 23])
@pytest.mark.parametrize("rows,classes,k", [(33, 1040, 2), (128, 4960, 4), (300, 1040, 2), (520, 4960, 4)])
def test_maxima_of_any_size(top, rows, classes, k):
    """A feature of `top` with a weight of one beside small whole numbers: every logit is exact in fp32.  The unit's exponential
    is good to 2^-22, as is a sum of them, and a softmax has three such factors (2^-20); its exponent x is rounded and so is
    the factor log2 e (2^-24 |x| each)."""
    g = torch.Generator().manual_seed(int(abs(top)) % 1000 + rows)
    feat = 72
    F = torch.randint(-1, 2, (rows, feat), generator=g).float() * (torch.rand(rows, feat, generator=g) < 0.2)
    W = torch.randint(-1, 2, (feat, classes), generator=g).float()
    F[:, 0], W[0] = top, 1.0
    labels = torch.randint(0, classes, (rows,), generator=g)
    Z = (F.double() @ W.double()).cuda()
    cut = lambda t, dim: [x.contiguous().cuda() for x in torch.tensor_split(t, k, dim)]
    f = sbp.SbpTensor((rows, feat), BF16, sbp.B, [F.to(BF16).cuda()] * k)
    w = sbp.SbpTensor((feat, classes), BF16, sbp.S(1), cut(W.to(BF16), 1))
    lab = sbp.SbpTensor((rows,), torch.int64, sbp.B, [labels.cuda()] * k)
    loss, m, s = (sbp.empty_global((rows,), F32, sbp.B, k, alias_replicas=True) for _ in range(3))
    ws = torch.empty(sbp.sbp_matmul_softmax_xent_workspace_bytes(f, w), dtype=torch.uint8, device="cuda")
    sbp.sbp_matmul_softmax_xent(f, w, lab, loss, m, s, ws)
    E = torch.exp(Z - Z.max(1, keepdim=True)[0])
    S = E.sum(1)
    assert torch.equal(m.locals[0].double(), Z.max(1)[0])
    assert float(((s.locals[0].double() - S) / S).abs().max()) <= 2.0 ** -21
    want = S.log() + (Z.max(1)[0] - Z[torch.arange(rows), labels.cuda()])
    assert float((loss.locals[0].double() - want).abs().max()) <= 2.0 ** -20 + 2.0 ** -23 * float(want.max())
    hit = torch.zeros(rows, classes, dtype=torch.bool, device="cuda")
    hit[torch.arange(rows), labels.cuda()] = True
    P = E / S[:, None]
    off = (2.0 ** -20 + 2.0 ** -23 * P.log2().abs()) * P
    for dtype, u in ((F32, 2.0 ** -24), (BF16, 2.0 ** -8)):      # half a unit of the result in its last place
        grad = sbp.empty_global((rows, classes), dtype, sbp.S(1), k)
        sbp.sbp_matmul_softmax_xent_backward(f, w, lab, m, s, grad)
        G = torch.cat(grad.locals, 1).double()
        assert bool(((G - P).abs() <= off + 1.01 * u * P)[~hit].all())
        assert bool(((G - (P - 1)).abs() <= off + 1.01 * u)[hit].all())
