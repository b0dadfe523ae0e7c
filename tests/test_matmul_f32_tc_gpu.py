"""fp32 products on the tensor cores where they can go wrong: edges of tiles and ring slots, chained segments of uneven
length, both stored forms of either operand, rows off the 16-byte rule, operands and sums that are not finite,
numbers at the ends of the exponent range.  The shapes are such as the library's own choice sends there (which
test_matmul_f32_forms_gpu.py checks, beside shapes that are forced).  Oracle and bound
as for the other fp32 products; the error against fp64 besides stays below what a chain of fp32 multiply-adds shows."""
import pytest
import torch

import paper_2110_15032_b200 as sbp
from test_ops_gpu import _matmul_case

pytestmark = pytest.mark.gpu
F32 = torch.float32
S0, S1, B = sbp.S(0), sbp.S(1), sbp.B


@pytest.mark.parametrize("M,K,N", [(1024, 1024, 512), (1027, 1029, 517), (513, 2047, 770), (640, 1500, 1039), (900, 992, 1155)])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, False), (False, True), (True, True)])
def test_edges_and_stored_forms(M, K, N, tx, tw):
    _matmul_case(M, K, N, 1, F32, B, B, tx=tx, tw=tw)


@pytest.mark.parametrize("M,K,N,k,xs,ws", [(1000, 1024, 1500, 4, S0, B), (1000, 1500, 777, 4, B, S1), (700, 1030, 900, 3, S0, B),
                                           (600, 1000, 1100, 7, B, S1)])
def test_groups(M, K, N, k, xs, ws):
    _matmul_case(M, K, N, k, F32, xs, ws)


@pytest.mark.parametrize("M,K,N,k", [(520, 2003, 640, 3), (768, 1100, 515, 8), (1030, 517, 900, 16)])
@pytest.mark.parametrize("ys", [B, S0, S1])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, True)])
def test_chained_segments(M, K, N, k, ys, tx, tw):
    _matmul_case(M, K, N, k, F32, S1, S0, ys=ys, tx=tx, tw=tw, flags=sbp.SBP_EPILOGUE_GELU if ys == S1 else 0)


def _product(X, W):
    (M, K), N = X.shape, W.shape[1]
    y = sbp.empty_global((M, N), F32, B, 1)
    sbp.sbp_matmul(sbp.SbpTensor((M, K), F32, B, [X]), sbp.SbpTensor((K, N), F32, B, [W]), y)
    return y.locals[0]


def _operands(M=1024, K=1024, N=640, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(M, K, device="cuda", generator=g), torch.randn(K, N, device="cuda", generator=g)


def _check(Y, X, W):
    R, mag = X.double() @ W.double(), X.double().abs() @ W.double().abs()
    fin = torch.isfinite(R) & (mag < 3e38)
    assert bool(((Y.double() - R).abs() <= 4 * X.shape[1] ** 0.5 * (2.0 ** -24 * mag + 2.0 ** -149))[fin].all())      # 2^-149: subnormal results
    return R, fin


def test_infinities_and_nan():
    X, W = _operands()
    X[3, 100], X[500, 7], X[1000, 1000] = float("inf"), -float("inf"), float("nan")
    W[5, 9], W[900, 600] = float("inf"), float("nan")
    Y = _product(X, W)
    R, fin = _check(Y, X, W)
    assert torch.equal(torch.isnan(Y), torch.isnan(R))
    assert torch.equal(Y[~fin & ~torch.isnan(R)].double(), R[~fin & ~torch.isnan(R)])


def test_ends_of_the_exponent_range():
    """The largest number is infinite once it is scaled; a sum may overflow; rows of small numbers and of large ones side by side."""
    X, W = _operands()
    X[7] *= 1e-30
    X[7, 20], W[20] = torch.finfo(F32).max, W[20] * 1e-30
    X[8], X[9], X[10] = X[8] * 1e30, X[9] * 2.0 ** -60, X[10] * 2.0 ** -100
    W[:, 5] *= 2.0 ** -40
    Y = _product(X, W)
    _check(Y, X, W)
    X[8, :2], W[:2, 6] = 3e38, 3.0
    assert bool(torch.isinf(_product(X, W)[8, 6]))


def test_whole_numbers_are_exact():
    g = torch.Generator(device="cuda").manual_seed(2)
    X = torch.randint(-90, 91, (1000, 1111), device="cuda", generator=g).float()
    W = torch.randint(-90, 91, (1111, 700), device="cuda", generator=g).float()
    assert torch.equal(_product(X, W).double(), X.double() @ W.double())


@pytest.mark.parametrize("M,K,N", [(1024, 512, 1024), (1000, 1500, 777), (2048, 2048, 512)])
def test_error_against_fp64(M, K, N):
    """A chain of K fp32 multiply-adds of independent normal numbers is off by about 0.21 sqrt(K / 2) 2^-23 of the result
    (2.8e-7 at 512, 5.6e-7 at 2048), a cut one by less in proportion to the root of the cut, at most eight."""
    X, W = _operands(M, K, N)
    R = X.double() @ W.double()
    err = float((_product(X, W).double() - R).norm() / R.norm())
    assert err <= 0.21 * (K / 16) ** 0.5 * 2.0 ** -23 + 6e-8


def test_the_same_bits_every_time():
    X, W = _operands(1000, 1500, 300)
    ref = _product(X, W).clone()
    for _ in range(20):
        assert torch.equal(ref, _product(X, W))


@pytest.mark.parametrize("M,K,N,k", [(1024, 1024, 640, 1), (300, 1029, 517, 3)])
@pytest.mark.parametrize("tx,tw", [(False, False), (True, False), (False, True), (True, True)])
def test_second_multiplication_edges(M, K, N, k, tx, tw):
    """One infinity in every row of X makes every tile be multiplied again: what is finite (columns where W is 0 there would be
    NaN, so W is not) is infinite, and with it out of the way of all but the first rows the others are ordinary results."""
    X, W = _operands(M, K, N)
    X[::128, 7] = float("inf")
    xl = [t.t().contiguous() if tx else t.contiguous() for t in torch.tensor_split(X, k, 1)]
    wl = [t.t().contiguous() if tw else t.contiguous() for t in torch.tensor_split(W, k, 0)]
    x = sbp.SbpTensor((K, M) if tx else (M, K), F32, S0 if tx else S1, xl)
    w = sbp.SbpTensor((N, K) if tw else (K, N), F32, S1 if tw else S0, wl)
    y = sbp.empty_global((M, N), F32, B, k)
    sbp.sbp_matmul_set_f32_form(sbp.SBP_F32_FORM_TENSOR)
    try:
        sbp.sbp_matmul(x, w, y, (sbp.SBP_TRANS_X if tx else 0) | (sbp.SBP_TRANS_W if tw else 0))
    finally:
        sbp.sbp_matmul_set_f32_form(sbp.SBP_F32_FORM_AUTO)
    Y = y.locals[0]
    _, fin = _check(Y, X, W)
    assert bool(fin[1:128].all()) and torch.equal(Y[::128], W[7].expand_as(Y[::128]).sign() * float("inf"))


def test_what_is_not_finite_costs_no_more_than_multiply_adds():
    """A tile is multiplied again at the rate of the multiply-add kernel: with every tile touched a product takes the sum of
    both, 4.5 to 6 times as long as on the tensor cores alone (chains of uncoalesced loads, as it once was, 140 times)."""
    X, W = _operands(1024, 1024, 1024)
    Xi = X.clone()
    Xi[::128, 7] = float("inf")
    times = []
    for a in (X, Xi):
        y = sbp.empty_global((1024, 1024), F32, B, 1)
        x, w = sbp.SbpTensor((1024, 1024), F32, B, [a]), sbp.SbpTensor((1024, 1024), F32, B, [W])
        for _ in range(3):
            sbp.sbp_matmul(x, w, y)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        for _ in range(20):
            sbp.sbp_matmul(x, w, y)
        t1.record()
        t1.synchronize()
        times.append(t0.elapsed_time(t1))
    assert times[1] < 12 * times[0], times


def _close(Y, X, W):
    """The bound of a chain of fp32 multiply-adds with nothing added but what subnormal numbers are rounded to; and as a whole the
    error of chains of K / 8 and their sum (0.21 sqrt(K / 16) 2^-23), the K roundings to 2^-149 being 0.29 of that each."""
    K = X.shape[1]
    R, mag = X.double() @ W.double(), X.double().abs() @ W.double().abs()
    assert bool(((Y.double() - R).abs() <= 4 * K ** 0.5 * 2.0 ** -24 * mag + 4 * K ** 0.5 * 2.0 ** -149).all())
    assert float((Y.double() - R).norm()) <= (0.21 * (K / 16) ** 0.5 * 2.0 ** -23 + 6e-8) * float(R.norm()) + K ** 0.5 / 3 * 2.0 ** -149 * R.numel() ** 0.5


def _scaled(T, e):
    """T 2^e by steps that lose nothing before the last."""
    while e < -120:
        T, e = T * 2.0 ** -120, e + 120
    return T * 2.0 ** e


@pytest.mark.parametrize("e", [-100, -108, -110, -112, -116, -120, -126, -130, -140])
@pytest.mark.parametrize("which", ["x", "w"])
def test_small_operands(e, which):
    """Numbers down to the subnormal ones, against others that make ordinary results of them."""
    X, W = _operands()
    X, W = (_scaled(X, e), W * 2.0 ** min(120, -e)) if which == "x" else (X * 2.0 ** min(120, -e), _scaled(W, e))
    _close(_product(X, W), X, W)


@pytest.mark.parametrize("e", [-105, -115, -126])
def test_some_small_operands(e):
    """Rows, columns and lone elements of them among ordinary ones, and results that lie wholly in the subnormal range."""
    X, W = _operands()
    X[::50], W[:, ::30] = _scaled(X[::50], e), W[:, ::30] * 2.0 ** 40
    X[5, ::3], W[::7, 4] = _scaled(X[5, ::3], e), _scaled(W[::7, 4], e)
    X[6] = 0.0
    X[6, 9], W[9] = 1.25 * 2.0 ** e * (1 + 2.0 ** -23), W[9] * 2.0 ** 60
    _close(_product(X, W), X, W)


@pytest.mark.parametrize("a,b", [(85, -85), (40, 9), (100, -100), (45, 45), (60, 2), (-60, -60), (-70, -60), (-40, -90), (-74, -74), (-20, -110)])
def test_results_of_any_size(a, b):
    """Small ones down to the subnormal, large operands and large sums."""
    X, W = _operands()
    X, W = X * 2.0 ** a, W * 2.0 ** b
    _close(_product(X, W), X, W)


@pytest.mark.parametrize("e", [-100, -112, -120, -126, -135, -145])
def test_a_permutation_moves_bits(e):
    X, _ = _operands(1024, 1024, 16)
    X = _scaled(X, e)
    order = torch.randperm(1024, generator=torch.Generator().manual_seed(3)).cuda()
    assert torch.equal(_product(X, torch.eye(1024, device="cuda")[order]), X[:, torch.argsort(order)])


def test_small_operands_that_do_not_matter():
    """Probabilities whose smallest are far below what the results can see."""
    _, W = _operands(1024, 1024, 1024)
    X = torch.softmax(torch.randn(1024, 1024, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5)) * 25, 1)
    assert int(((X > 0) & (X < 2.0 ** -110)).sum()) > 1000
    _close(_product(X, W), X, W)
