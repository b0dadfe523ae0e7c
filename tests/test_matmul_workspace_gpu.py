"""The two workspace queries of a product: the larger one's size alone makes a long contraction be cut over the device, a
product for which both answer the same leaves a larger workspace alone, and cutting K (over the pairs of a cluster, or over
clusters) is no further from fp64 than one accumulator over all of it."""
import pytest
import torch

import paper_2110_15032_b200 as sbp

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16
S0, S1, B = sbp.S(0), sbp.S(1), sbp.B


def _product(M, K, N, k, ys, out_dtype, seed=7):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(M, K, generator=g, device="cuda").to(BF16)
    W = (torch.randn(K, N, generator=g, device="cuda") / K ** 0.5).to(BF16)
    x = sbp.SbpTensor((M, K), BF16, S1, [t.contiguous() for t in torch.tensor_split(X, k, 1)])
    w = sbp.SbpTensor((K, N), BF16, S0, [t.contiguous() for t in torch.tensor_split(W, k, 0)])
    return x, w, sbp.empty_global((M, N), out_dtype, ys, k), X.double() @ W.double()


def _whole(y):
    return y.locals[0].double() if y.sig == B else torch.cat([t.double() for t in y.locals], y.sig.axis)


@pytest.mark.parametrize("M,K,N,k,ys", [(64, 131072, 256, 8, B), (512, 262144, 512, 8, B), (130, 100000, 256, 2, S0), (40, 100003, 72, 1, B)])
def test_the_queried_room_is_used(M, K, N, k, ys):
    x, w, y, _ = _product(M, K, N, k, ys, BF16)
    least, preferred = sbp.sbp_matmul_workspace_bytes(x, w, y), sbp.sbp_matmul_workspace_bytes_preferred(x, w, y)
    assert preferred >= least + 2 * 4 * M * N
    launches, split = [], []
    for n in (least, preferred):
        ws = torch.empty(max(256, n), dtype=torch.uint8, device="cuda")
        before, s = sbp.sbp_launch_count(), sbp.sbp_matmul_split_launches()
        sbp.sbp_matmul(x, w, y, 0, ws)
        launches.append(sbp.sbp_launch_count() - before)
        split.append(sbp.sbp_matmul_split_launches() - s)
    torch.cuda.synchronize()
    assert launches[1] == launches[0] + 1 and split[1] == 1


@pytest.mark.parametrize("M,K,N,k", [(512, 1024, 2048, 4), (16, 4096, 4096, 8), (2048, 2048, 2048, 1), (333, 333, 333, 3)])
def test_a_workspace_without_a_use_is_left_alone(M, K, N, k):
    x, w, y, _ = _product(M, K, N, k, B, BF16)
    least = sbp.sbp_matmul_workspace_bytes(x, w, y)
    assert least == sbp.sbp_matmul_workspace_bytes_preferred(x, w, y)
    ws = torch.full((64 << 20,), 0xAB, dtype=torch.uint8, device="cuda")
    sbp.sbp_matmul(x, w, y, 0, ws)
    assert bool((ws[least:] == 0xAB).all())


@pytest.mark.parametrize("M,K,N,k", [(16, 16384, 4096, 8), (64, 131072, 256, 8), (512, 65536, 512, 8), (1000, 4096, 1024, 4), (33, 1000, 520, 1)])
def test_cutting_k_is_no_further_from_fp64(M, K, N, k):
    """fp32 results; the uncut form sums all of K in one accumulator, as every product did before the split form."""
    x, w, y, ref = _product(M, K, N, k, B, F32)
    ws = torch.empty(max(256, sbp.sbp_matmul_workspace_bytes_preferred(x, w, y)), dtype=torch.uint8, device="cuda")
    off = {}
    try:
        for name, form, room in (("uncut", sbp.SBP_TC_FORM_SQUARE, None), ("split", sbp.SBP_TC_FORM_SPLIT, None), ("chosen", sbp.SBP_TC_FORM_AUTO, ws)):
            sbp.sbp_matmul_set_form(form, 0)
            sbp.sbp_matmul(x, w, y, 0, room)
            off[name] = float((_whole(y) - ref).norm() / ref.norm())
    finally:
        sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_AUTO, 0)
    # 5 %: where both are a few roundings of the last bit the two norms differ by chance
    assert max(off["split"], off["chosen"]) <= 1.05 * off["uncut"], off
