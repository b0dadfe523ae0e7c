"""Row sums of the split softmax against fp64: no further off than one unit in the last place (2^-23, root mean square over
the rows), whatever the spread of the logits, the length of the rows and the kernel that takes them; and masks of the
type's lowest value count as nothing.  An exponential is good to 2^-22 and 5e-8 low on the average; what is added to that --
the exponent's rounding, the changes of maximum inside a thread, between threads and between parts -- has to stay below it."""
import pytest
import torch

import paper_2110_15032_b200 as sbp

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


def _forward(Z, k):
    rows, classes = Z.shape
    z = sbp.SbpTensor((rows, classes), Z.dtype, sbp.S(1), [t.contiguous() for t in torch.tensor_split(Z, k, 1)])
    lab = sbp.SbpTensor((rows,), torch.int64, sbp.B, [torch.zeros(rows, dtype=torch.int64, device="cuda")] * k)
    loss, m, s = (sbp.empty_global((rows,), F32, sbp.B, k) for _ in range(3))
    ws = torch.empty(max(4, sbp.sbp_softmax_xent_workspace_bytes(z)), dtype=torch.uint8, device="cuda")
    sbp.sbp_softmax_xent(z, lab, loss, m, s, ws)
    return loss.locals[0], m.locals[0], s.locals[0]


@pytest.mark.parametrize("rows,classes,k,dtype,std", [
    (20000, 100, 4, F32, 2), (5000, 100, 4, BF16, 2), (740, 10000, 8, BF16, 2), (740, 10000, 8, F32, 8), (3000, 4096, 4, F32, 2),
    (700, 10000, 8, F32, 2), (256, 100003, 4, F32, 2), (256, 100003, 4, F32, 20), (700, 100003, 4, BF16, 2), (700, 130, 2, F32, 30)])
def test_row_sums(rows, classes, k, dtype, std):
    g = torch.Generator(device="cuda").manual_seed(classes)
    Z = torch.empty(rows, classes, device="cuda").normal_(0.0, std, generator=g).to(dtype)
    _, m, s = _forward(Z, k)
    Zd = Z.double()
    want = torch.exp(Zd - Zd.max(1, keepdim=True)[0]).sum(1)
    assert torch.equal(m.double(), Zd.max(1)[0])
    assert float(((s.double() - want) / want).square().mean().sqrt()) <= 2.0 ** -23


@pytest.mark.parametrize("rows,classes,k", [(5, 70, 2), (300, 20000, 2), (800, 1000, 3), (3000, 257, 1), (40, 33, 4)])
@pytest.mark.parametrize("dtype", [F32, BF16])
def test_masked_classes_count_as_nothing(rows, classes, k, dtype):
    """Whole threads' shares masked, every second class masked, and -inf beside the lowest value."""
    g = torch.Generator(device="cuda").manual_seed(rows)
    Z = torch.empty(rows, classes, device="cuda").normal_(0.0, 2.0, generator=g).to(dtype)
    keep = Z.clone()
    low = torch.finfo(dtype).min
    Z[:, classes // 2:] = low
    Z[:, 1::2] = low
    Z[:, 3] = -float("inf")
    keep[:, classes // 2:] = -float("inf")
    keep[:, 1::2] = -float("inf")
    loss, m, s = _forward(Z, k)
    want = torch.nn.functional.cross_entropy(keep.double(), torch.zeros(rows, dtype=torch.int64, device="cuda"), reduction="none")
    assert torch.equal(m.double(), keep.double().max(1)[0])
    assert torch.allclose(loss.double(), want, rtol=1e-6, atol=1e-6)


def test_infinities_and_nan_reach_the_loss():
    Z = torch.randn(900, 500, device="cuda")
    Z[7, 100], Z[8, 499], Z[9, 3] = float("nan"), float("inf"), -float("inf")
    Z = torch.cat([Z, Z[:20]], 0)
    for part in (Z, Z[:100].contiguous()):
        loss = _forward(part, 2)[0]
        bad = torch.isnan(loss) | torch.isinf(loss)
        assert bool(bad[7]) and bool(bad[8]) and not bool(bad[9]) and int(bad[:100].sum()) == 2


@pytest.mark.parametrize("top", [3e4, 1e6, -3e4, -1e8, -1e9, -1e10, -1e20, -1e30, None])
@pytest.mark.parametrize("rows,classes,k", [(40, 1000, 2), (300, 20001, 4), (4000, 515, 2)])
@pytest.mark.parametrize("dtype", [F32, BF16])
def test_maxima_of_any_size(top, rows, classes, k, dtype):
    """Rows wholly at one value, as a padded row under a mask is: the sum is the class count and the gradient 1 / classes; and
    the same rows with half of their classes lower by a few units in the last place, or by ln 2 where those are finer."""
    v = torch.tensor(torch.finfo(dtype).min if top is None else top, dtype=dtype, device="cuda")
    Z = v.expand(rows, classes).clone()
    step = max(0.6931471805599453, float(v.abs()) * 2.0 ** (-22 if dtype == F32 else -6))
    Z[rows // 2:, ::2] = v.float() * 1.0 - step if top is not None else v
    Zd = Z.double()
    E = torch.exp(Zd - Zd.max(1, keepdim=True)[0])
    want = E.sum(1)
    loss, m, s = _forward(Z, k)
    assert torch.equal(m.double(), Zd.max(1)[0])
    assert float(((s.double() - want) / want).abs().max()) <= 2.0 ** -21
    gone = Zd.max(1)[0] - Zd[:, 0]
    assert bool(((loss.double() - want.log() - gone).abs() <= 2.0 ** -20 + 2.0 ** -23 * gone).all())
    z = sbp.SbpTensor((rows, classes), dtype, sbp.S(1), [t.contiguous() for t in torch.tensor_split(Z, k, 1)])
    lab = sbp.SbpTensor((rows,), torch.int64, sbp.B, [torch.zeros(rows, dtype=torch.int64, device="cuda")] * k)
    rm, rs = (sbp.SbpTensor((rows,), F32, sbp.B, [t] * k) for t in (m, s))
    g = sbp.empty_global((rows, classes), dtype, sbp.S(1), k)
    sbp.sbp_softmax_xent_backward(z, lab, rm, rs, g)
    G = torch.cat(g.locals, 1).double()
    # three factors good to 2^-22, an exponent x rounded to 2^-24 |x| and as much from log2 e, the result's own rounding; what
    # is below the smallest normal number becomes 0
    u = 2.0 ** -24 if dtype == F32 else 2.0 ** -8
    P = E / want[:, None]
    off = (2.0 ** -20 + 2.0 ** -23 * P.clamp(min=2.0 ** -126).log2().abs()) * P + 2.0 ** -126
    assert bool(((G - P).abs() <= off + 1.01 * u * P)[:, 1:].all())
    assert bool(((G - (P - 1.0)).abs() <= off + 1.01 * u)[:, 0].all())
