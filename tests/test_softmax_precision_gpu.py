"""Row sums of the split softmax for many rows of many classes, at every team the library takes and where it leaves rows
to the partial kernel.  Bound: an element's exponent has the rounding of one fma, at most 2^-24 |z - m| log2 e, and its
ex2 is good to 2^-22, both of which average out over a row; what a whole thread shares (one change of units, the merges)
is a few ex2: 1e-6 relative, a fifth of what the carried sums lost when every chunk scaled them."""
import pytest
import torch

import paper_2110_15032_b200 as sbp

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


@pytest.mark.parametrize("rows,classes,k,dtype", [(3000, 8191, 2, F32), (3000, 8193, 2, F32), (1480, 16384, 3, F32), (1479, 32768, 2, F32),
                                                  (740, 33100, 3, F32), (2960, 32768, 4, BF16), (1000, 66000, 2, BF16), (739, 9000, 4, F32)])
def test_row_sums(rows, classes, k, dtype):
    g = torch.Generator(device="cuda").manual_seed(rows)
    Z = torch.empty(rows, classes, device="cuda").normal_(0.0, 2.0, generator=g).to(dtype)
    z = sbp.SbpTensor((rows, classes), dtype, sbp.S(1), [t.contiguous() for t in torch.tensor_split(Z, k, 1)])
    lab = sbp.SbpTensor((rows,), torch.int64, sbp.B, [torch.randint(0, classes, (rows,), device="cuda", generator=g)] * k)
    loss, m, S = (sbp.empty_global((rows,), F32, sbp.B, k) for _ in range(3))
    ws = torch.empty(sbp.sbp_softmax_xent_workspace_bytes(z), dtype=torch.uint8, device="cuda")
    sbp.sbp_softmax_xent(z, lab, loss, m, S, ws)
    Zd = Z.double()
    mx = Zd.max(1)[0]
    want = torch.exp(Zd - mx[:, None]).sum(1)
    assert torch.equal(m.locals[0].double(), mx)
    assert float(((S.locals[0].double() - want) / want).abs().max()) <= 1e-6
