"""Narrow bases (k + r <= 128) on contiguous bf16 matrices of odd width: the tensor-core products that take the
rows in classes, at remainders of classes, tiles and K steps.

Z is compared with the exact product of the same operands rounded to bf16 (the basis enters as fp32): half a
unit in the last place, 2^-9, plus what the fp32 sums may move across a rounding boundary.  The gradient is
compared with the exact one from the same Z: fp32 sums over the tokens (a random walk of sqrt(N) 2^-24, some
digits more for the order of the pieces) and an fp32 product."""
import pytest
import torch

from paper_2602_23111_b200 import api

pytestmark = pytest.mark.gpu


def _basis(d, k, r, c, g):
    P = torch.linalg.qr(torch.randn(d, k + r, generator=g, device="cuda", dtype=torch.float64))[0].float()
    b = api.Basis(d, k, r, torch.bfloat16)
    b.set(P[:, :k].contiguous(), P[:, k:].contiguous(), c)
    return b, P


@pytest.mark.parametrize("N,d,k,r,d_out", [
    (129, 259, 8, 8, 131), (513, 257, 40, 24, 511), (2047, 1179, 37, 37, 1251), (4100, 1022, 64, 64, 2050), (20001, 5461, 63, 64, 901),
    (3000, 780, 3, 1, 1004), (2500, 771, 0, 31, 333), (1500, 333, 65, 62, 4001),
])
def test_products_with_rows_taken_in_classes(N, d, k, r, d_out):
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    X = torch.randn(N, d, generator=g, device="cuda").bfloat16()
    dY = torch.randn(N, d_out, generator=g, device="cuda").bfloat16()
    c, s = 2.5, k + r
    b, P = _basis(d, k, r, c, g)
    wide = torch.full((N, (s + 7) // 8 * 8 + 8), 7.0, device="cuda", dtype=torch.bfloat16)
    Z = b.compress(X, out=wide[:, :s])
    assert bool((wide[:, s:] == 7.0).all())
    Z64 = X.double() @ P.double()
    err = (Z.double() - Z64).abs()
    assert bool((err <= Z64.abs() * 2 ** -8 + 1e-4).all())
    assert float((Z.double() - Z64).norm() / Z64.norm()) <= 2e-3       # uniform rounding: 2^-9 / sqrt(3) and less
    M = b.weight_grad_partial(dY, Z)
    M64 = dY.double().t() @ Z.double()
    assert float((M.double() - M64).norm() / M64.norm()) <= 5e-5
    M64[:, k:] *= c
    dW64 = M64 @ P.double().t()
    for base in (None, torch.ones(d_out, d, device="cuda")):
        dW = b.weight_grad(dY, Z, out=None if base is None else base.clone(), accumulate=base is not None)
        got = dW.double() - (0 if base is None else base.double())
        worst = (got - dW64).norm(dim=1) / dW64.norm(dim=1)
        assert float((got - dW64).norm() / dW64.norm()) <= 5e-5 and float(worst.max()) <= 5e-4
    assert torch.equal(b.compress(X), Z)
    assert b.status() == api.PRAC_OK


def test_scratch_of_the_aligned_layout_is_still_enough():
    # a caller that brings only what an aligned dY needs gets the general path, the same numbers to fp32 rounding
    g = torch.Generator(device="cuda")
    g.manual_seed(12)
    N, d, k, r, d_out = 3001, 515, 24, 16, 777
    X = torch.randn(N, d, generator=g, device="cuda").bfloat16()
    dY = torch.randn(N, d_out, generator=g, device="cuda").bfloat16()
    b, _ = _basis(d, k, r, 1.5, g)
    Z = b.compress(X)
    want = b.weight_grad(dY, Z)
    ws = torch.empty(d_out * (k + r) * 4 + 256 + b.grad_workspace_bytes(N, 776), dtype=torch.uint8, device="cuda")
    got = b.weight_grad(dY, Z, ws=ws)
    assert float((got - want).norm() / want.norm()) <= 5e-5
    # and a base pointer off the grid
    Xo = torch.empty(N * d + 1, dtype=torch.bfloat16, device="cuda")[1:].view(N, d)
    Xo.copy_(X)
    Zo = b.compress(Xo)
    assert float((Zo.double() - Z.double()).norm() / Z.double().norm()) <= 1e-4


@pytest.mark.parametrize("N,d,ld,k,r", [
    (300, 259, 259, 32, 32), (300, 259, 261, 32, 32), (4099, 1179, 1179, 64, 64), (2047, 1179, 1211, 37, 36), (130, 131, 133, 3, 0),
    (300, 259, 261, 96, 96), (1030, 1179, 1182, 300, 301),
])
def test_what_is_not_finite_stays_in_its_own_row(N, d, ld, k, r):
    # ld > d: the elements between the rows are NaN, and no part of X
    g = torch.Generator(device="cuda")
    g.manual_seed(13)
    b, P = _basis(d, k, r, 1.5, g)
    buf = torch.full((N, ld), float("nan"), device="cuda", dtype=torch.bfloat16)
    X = buf[:, :d]
    X.copy_(torch.randn(N, d, generator=g, device="cuda"))
    clean = b.compress(X.contiguous() if ld == d else X)
    assert bool(torch.isfinite(clean).all())
    assert float((clean.double() - X.double() @ P.double()).norm() / clean.double().norm()) <= 5e-3
    if k + r > 128:
        return                      # (contiguous: finite numbers throughout, by the interface)
    bad = {0: float("inf"), 5: float("nan"), N // 2: float("-inf"), N - 1: float("inf")}
    for row, v in bad.items():
        X[row, (7 * row) % d] = v
    Z = b.compress(X)
    want = X.double() @ P.double()
    rows = torch.tensor(sorted(bad), device="cuda")
    rest = torch.ones(N, dtype=torch.bool, device="cuda")
    rest[rows] = False
    assert torch.equal(Z[rest], clean[rest])
    assert torch.equal(Z[rows].double(), want[rows]) or bool((torch.isnan(Z[rows]) == torch.isnan(want[rows])).all()
                                                             and (Z[rows].double().nan_to_num(7.0) == want[rows].nan_to_num(7.0)).all())
