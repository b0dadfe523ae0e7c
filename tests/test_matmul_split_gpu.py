"""The split form of the tensor-core MatMul where it can go wrong: ragged edges of its tiles, tiles and
contractions shorter than a group of K-blocks, segments of uneven and zero length, exchanged operands,
results the vector stores cannot address, replicas, and that the library's own choice takes it.
Oracle and tolerance (2e-2 relative, 1e-3 absolute against fp64) as for the other bf16 products."""
import pytest
import torch

import paper_2110_15032_b200 as sbp
from test_ops_gpu import _matmul_case

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16
S0, S1, B, P = sbp.S(0), sbp.S(1), sbp.B, sbp.P_SUM


@pytest.fixture
def split():
    sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_SPLIT, 0)
    yield
    sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_AUTO, 0)


# one row to several tiles of either orientation; one K-block to enough for every split; edges off by one
@pytest.mark.parametrize("M", [1, 15, 33, 64, 129, 257, 500])
@pytest.mark.parametrize("K,N", [(40, 72), (64, 256), (136, 264), (1000, 520), (2056, 1032)])
@pytest.mark.parametrize("tw", [False, True])
def test_sizes(split, M, K, N, tw):
    _matmul_case(M, K, N, 1, BF16, B, B, tw=tw, flags=sbp.SBP_EPILOGUE_GELU if M == 33 else 0)
    _matmul_case(M, K, N, 3, BF16, B, S1, tw=tw, out_dtype=F32 if M == 64 else BF16)


@pytest.mark.parametrize("M,K,N", [(64, 200, 72), (264, 1000, 520), (520, 16, 136)])
def test_transposed_rows(split, M, K, N):
    _matmul_case(M, K, N, 2, BF16, S1, S0, ys=B, tx=True)
    _matmul_case(M, K, N, 1, BF16, B, B, tx=True, tw=True, out_dtype=F32)


@pytest.mark.parametrize("M,K,N,k", [(40, 1048, 136, 8), (100, 3, 72, 8), (20, 5000, 80, 3), (300, 808, 264, 3)])
@pytest.mark.parametrize("ys", [B, S0, S1])
def test_chained_segments_and_replicas(split, M, K, N, k, ys):
    _matmul_case(M, K, N, k, BF16, S1, S0, ys=ys, flags=sbp.SBP_EPILOGUE_GELU if ys == S0 else 0, out_dtype=F32)


def test_results_the_vector_stores_cannot_address(split):
    _matmul_case(17, 512, 333, 2, BF16, B, B)
    _matmul_case(200, 512, 333, 2, BF16, B, S1)


@pytest.mark.parametrize("M,K,N,k,ys", [(40, 100000, 72, 1, B), (264, 80001, 136, 8, B), (16, 200000, 100, 3, S1), (130, 100000, 255, 2, S0)])
@pytest.mark.parametrize("out_dtype", [BF16, F32])
def test_contraction_cut_over_many_clusters(split, M, K, N, k, ys, out_dtype):
    """With room in the workspace for several copies of the result; replicas, GeLU, columns that 4 does not divide."""
    torch.manual_seed(5)
    X, W = torch.randn(M, K, device="cuda").to(BF16), (torch.randn(K, N, device="cuda") / K ** 0.5).to(BF16)
    xl = [t.contiguous() for t in torch.tensor_split(X, k, 1)]
    wl = [t.contiguous() for t in torch.tensor_split(W, k, 0)]
    x, w = sbp.SbpTensor((M, K), BF16, S1, xl), sbp.SbpTensor((K, N), BF16, S0, wl)
    y = sbp.empty_global((M, N), out_dtype, ys, k)
    flags = sbp.SBP_EPILOGUE_GELU if N == 100 else 0
    need = sbp.sbp_matmul_workspace_bytes(x, w, y, flags)
    few = torch.empty(max(16, need), dtype=torch.uint8, device="cuda")
    room = torch.empty(need + 40 * M * (N + 3) * 4, dtype=torch.uint8, device="cuda")
    ref = X.double() @ W.double()
    ref = torch.nn.functional.gelu(ref) if flags else ref
    before = sbp.sbp_launch_count()
    sbp.sbp_matmul(x, w, y, flags, few)
    once = sbp.sbp_launch_count() - before
    for _ in range(2):
        for t in y.locals:
            t.fill_(float("nan"))
        before = sbp.sbp_launch_count()
        sbp.sbp_matmul(x, w, y, flags, room)
        assert sbp.sbp_launch_count() - before == once + 1, "the partial results are added up by a kernel of their own"
        got = y.locals[0].double() if ys == B else torch.cat([t.double() for t in y.locals], 0 if ys == S0 else 1)
        assert bool(((got - ref).abs() <= 1e-3 + 2e-2 * ref.abs()).all())
        if ys == B:
            assert all(torch.equal(y.locals[0], t) for t in y.locals)


def test_the_library_takes_the_split_form_for_few_tiles():
    """The same bits every time, and far fewer operand tiles than CTA pairs so that the choice is clear."""
    X, W = torch.randn(16, 8192, device="cuda").to(BF16), torch.randn(8192, 1024, device="cuda").to(BF16)
    x, w = sbp.SbpTensor((16, 8192), BF16, B, [X]), sbp.SbpTensor((8192, 1024), BF16, B, [W])
    y = sbp.empty_global((16, 1024), BF16, B, 1)
    sbp.sbp_matmul(x, w, y)
    ref = y.locals[0].clone()
    for _ in range(20):
        sbp.sbp_matmul(x, w, y)
        assert torch.equal(ref, y.locals[0])
    sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_SPLIT, 0)
    try:
        sbp.sbp_matmul(x, w, y)
        assert torch.equal(ref, y.locals[0]), "the automatic choice is the split form's"
    finally:
        sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_AUTO, 0)
