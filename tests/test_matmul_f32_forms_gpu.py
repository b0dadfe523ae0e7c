"""The three kernels of fp32 products, each forced and each counted: edges of its tiles and K-slices, contractions of one slice and
of many a warp, chained segments of uneven and zero length, both stored forms, more tiles than the early release of the small
kernel allows.  And what the library picks by itself, where the other tests of these kernels rely on it."""
import time

import pytest
import torch

import paper_2110_15032_b200 as sbp
from test_ops_gpu import _matmul_case

pytestmark = pytest.mark.gpu
F32 = torch.float32
S0, S1, B = sbp.S(0), sbp.S(1), sbp.B
TILED, SMALL, TENSOR = sbp.SBP_F32_FORM_TILED, sbp.SBP_F32_FORM_SMALL, sbp.SBP_F32_FORM_TENSOR


@pytest.fixture(autouse=True)
def _the_librarys_choice_afterwards():
    yield
    sbp.sbp_matmul_set_f32_form(sbp.SBP_F32_FORM_AUTO)


def _case(form, *args, **kw):
    """One product on the kernel `form`, forced or (0) as chosen; returns the kernel that ran."""
    sbp.sbp_matmul_set_f32_form(form)
    before = sbp.sbp_matmul_f32_form_stats()
    _matmul_case(*args, **kw)
    ran = [b - a for a, b in zip(before, sbp.sbp_matmul_f32_form_stats())]
    assert sum(ran) == 1 and (not form or ran[form - 1] == 1), (form, ran)
    return ran.index(1) + 1


@pytest.mark.parametrize("M,K,N", [(2048, 64, 2048), (1153, 37, 2050), (512, 256, 512), (500, 250, 509),      # 128 x 128, the latter cut in eight
                                   (64, 16, 64), (65, 17, 63), (40, 2500, 24), (257, 130, 1030)])               # 64 x 64
@pytest.mark.parametrize("tx,tw", [(False, False), (True, True)])
def test_tiled(M, K, N, tx, tw):
    _case(TILED, M, K, N, 1, F32, B, B, tx=tx, tw=tw)


@pytest.mark.parametrize("K", [1, 16, 17, 127, 129, 260, 1000])
@pytest.mark.parametrize("M,N", [(1, 1), (33, 65), (100, 36), (31, 200), (225, 131)])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, False), (False, True), (True, True)])
def test_small(M, K, N, tx, tw):
    _case(SMALL, M, K, N, 1, F32, B, B, tx=tx, tw=tw)


@pytest.mark.parametrize("K", [1, 31, 33, 64, 257])
@pytest.mark.parametrize("M,N", [(1, 1), (128, 16), (129, 17), (127, 193), (130, 400)])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, False), (False, True), (True, True)])
def test_tensor(M, K, N, tx, tw):
    _case(TENSOR, M, K, N, 1, F32, B, B, tx=tx, tw=tw)


@pytest.mark.parametrize("form", [TILED, SMALL, TENSOR])
@pytest.mark.parametrize("M,K,N,k", [(70, 45, 83, 3), (33, 5, 130, 8), (200, 700, 90, 5)])
@pytest.mark.parametrize("ys", [B, S0, S1])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, True)])
def test_groups_and_segments(form, M, K, N, k, ys, tx, tw):
    _case(form, M, K, N, k, F32, S0, B, tx=tx, tw=tw)
    _case(form, M, K, N, k, F32, B, S1, tx=tx, tw=tw)
    _case(form, M, K, N, k, F32, S1, S0, ys=ys, tx=tx, tw=tw, flags=sbp.SBP_EPILOGUE_GELU if ys == S0 else 0)


def test_the_librarys_choice():
    """Far from the lines between them: tests of the tensor cores' accuracy and of its ranges count on this one."""
    assert _case(0, 64, 128, 96, 2, F32, S0, B) == SMALL
    assert _case(0, 32, 512, 32, 1, F32, B, B) == TILED
    assert _case(0, 1155, 124, 1248, 3, F32, B, S1) != SMALL      # ten CTAs an SM: 20.7 us, tiled 17.2, tensor cores 12.6
    for M, K, N in ((1024, 1024, 640), (1000, 1500, 777), (1000, 1111, 700), (1024, 512, 1024), (2048, 2048, 512), (1000, 1500, 300)):
        assert _case(0, M, K, N, 1, F32, B, B) == TENSOR


@pytest.mark.parametrize("M,K,N", [(87, 66, 334), (185, 67, 678), (99, 100, 70), (300, 130, 90), (64, 400, 96)])
def test_small_is_no_further_off_than_tiled(M, K, N):
    """Root mean square over the results, operands of one sign, whose roundings all show; 1 %: what two draws differ by."""
    g = torch.Generator(device="cuda").manual_seed(K)
    X, W = torch.randn(M, K, device="cuda", generator=g).abs(), torch.randn(K, N, device="cuda", generator=g).abs()
    R, off = X.double() @ W.double(), {}
    for form in (TILED, SMALL):
        y = sbp.empty_global((M, N), F32, B, 1)
        sbp.sbp_matmul_set_f32_form(form)
        sbp.sbp_matmul(sbp.SbpTensor((M, K), F32, B, [X]), sbp.SbpTensor((K, N), F32, B, [W]), y)
        off[form] = float((y.locals[0].double() - R).norm())
    assert off[SMALL] <= 1.01 * off[TILED]


def test_the_search_for_a_cut_is_cheap_on_the_host():
    """What a call costs the host on the tensor cores, whose tile width and cut are searched for, against the tiled kernel: 1.05
    times as much (1.5 times where the search asked the device its number 78 times)."""
    k, M, K, N = 8, 1000, 1024, 1500
    x = sbp.SbpTensor((M, K), F32, S0, [t.contiguous() for t in torch.tensor_split(torch.randn(M, K, device="cuda"), k, 0)])
    w = sbp.SbpTensor((K, N), F32, B, [torch.randn(K, N, device="cuda")] * k)
    y = sbp.empty_global((M, N), F32, S0, k)
    least = {TILED: 1e9, TENSOR: 1e9}
    for _ in range(30):
        for form in least:
            sbp.sbp_matmul_set_f32_form(form)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(20):
                sbp.sbp_matmul(x, w, y)
            least[form] = min(least[form], time.perf_counter() - t0)
    torch.cuda.synchronize()
    assert least[TENSOR] < 1.3 * least[TILED], least
