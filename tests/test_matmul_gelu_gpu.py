"""GeLU in the epilogue of the tensor-core products, number by number: a contraction of one with ones leaves W itself."""
import hashlib
import os

import pytest
import torch

import paper_2110_15032_b200 as sbp

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


@pytest.mark.parametrize("form", [sbp.SBP_TC_FORM_SQUARE, sbp.SBP_TC_FORM_TALL, sbp.SBP_TC_FORM_SPLIT])
@pytest.mark.parametrize("out", [F32, BF16])
def test_gelu_of_every_kind_of_number(form, out):
    """Approximation 7.1.26 is good to 1.5e-7 in erf, half of that times |v| here; its special functions, its rounded constants
    and the roundings of the sum add a few units in the last place of |v| (2^-22 |v|), a bf16 result its own."""
    M, N = 300, 2048
    v = torch.cat([torch.linspace(-12, 12, N - 16, device="cuda"), torch.tensor(
        [0.0, -0.0, 1e-30, -1e-30, 3e-3, -3e-3, 31.5, -31.5, 40.0, -40.0, 1e30, -1e30, 3e38, -3e38, float("inf"), float("nan")],
        device="cuda")]).to(BF16)
    X, W = torch.ones(M, 1, dtype=BF16, device="cuda"), v[None, :].contiguous()
    x, w = sbp.SbpTensor((M, 1), BF16, sbp.B, [X]), sbp.SbpTensor((1, N), BF16, sbp.B, [W])
    y = sbp.empty_global((M, N), out, sbp.B, 1)
    ws = torch.empty(max(256, sbp.sbp_matmul_workspace_bytes(x, w, y, sbp.SBP_EPILOGUE_GELU)), dtype=torch.uint8, device="cuda")
    sbp.sbp_matmul_set_form(form, 0)
    try:
        sbp.sbp_matmul(x, w, y, sbp.SBP_EPILOGUE_GELU, ws)
    finally:
        sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_AUTO, 0)
    got, vd = y.locals[0].double(), v.double()
    assert bool(torch.isnan(got[:, -1]).all()) and bool(torch.isposinf(got[:, -2]).all())
    want = 0.5 * vd * torch.special.erfc(-vd / 2 ** 0.5)
    tol = vd.abs() * (0.75e-7 + 2.0 ** -22) + (want.abs() * 2.0 ** -8 if out == BF16 else 0.0) + 1e-37
    assert bool(((got - want).abs() <= tol)[:, :-2].all())


@pytest.mark.parametrize("form", [sbp.SBP_TC_FORM_SQUARE, sbp.SBP_TC_FORM_TALL, sbp.SBP_TC_FORM_SPLIT])
@pytest.mark.parametrize("out", [F32, BF16])
def test_gelu_keeps_its_bits(form, out):
    """The formula's operations in the formula's order, whichever way they are issued: a program's results do not move."""
    v = torch.arange(1 << 16, dtype=torch.int32, device="cuda").to(torch.int16).view(BF16)
    X = torch.ones(300, 1, dtype=BF16, device="cuda")
    x, w = sbp.SbpTensor((300, 1), BF16, sbp.B, [X]), sbp.SbpTensor((1, 1 << 16), BF16, sbp.B, [v[None, :].contiguous()])
    y = sbp.empty_global((300, 1 << 16), out, sbp.B, 1)
    ws = torch.empty(max(256, sbp.sbp_matmul_workspace_bytes(x, w, y, sbp.SBP_EPILOGUE_GELU)), dtype=torch.uint8, device="cuda")
    sbp.sbp_matmul_set_form(form, 0)
    try:
        sbp.sbp_matmul(x, w, y, sbp.SBP_EPILOGUE_GELU, ws)
    finally:
        sbp.sbp_matmul_set_form(sbp.SBP_TC_FORM_AUTO, 0)
    Y = y.locals[0].cpu()
    Y[torch.isnan(Y)] = float("nan")
    bits = Y.view(torch.int32 if out == F32 else torch.int16)
    assert bool((bits == bits[0]).all())
    with open(os.path.join(os.path.dirname(__file__), "golden", "gelu_of_every_bf16.txt")) as f:
        golden = dict(line.split() for line in f if not line.startswith("#"))
    assert hashlib.sha256(bits[0].numpy().tobytes()).hexdigest() == golden["f32" if out == F32 else "bf16"]
