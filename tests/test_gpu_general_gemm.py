"""The general FMA product behind fp32 storage, at the edges of its tiles and of its K pieces, through the
entry points that reach it: every operand order, aligned and unaligned rows, the accumulated and the
symmetric output.

Bound: an fp32 sum of K products differs from the exact one by at most K 2^-24 (relative to the sum of the
absolute products); for random signs the error of the matrix is about sqrt(K) 2^-24 of its norm, and the
pieces K is cut into only shorten the chains.  4 sqrt(K) 2^-24 + 2^-22 covers it."""
import math

import pytest
import torch

from paper_2602_23111_b200 import api

pytestmark = pytest.mark.gpu


def _close(got, want, K, what):
    want = want.double()
    err = (got.double() - want).norm() / want.norm()
    worst = (got.double() - want).norm(dim=1) / want.norm(dim=1).clamp_min(1e-300)
    bound = 4 * math.sqrt(K) * 2 ** -24 + 2 ** -22
    assert err <= bound, (what, float(err), bound)
    assert worst.max() <= 8 * bound, (what, float(worst.max()))


def _rows(n, cols, pad, g):
    return torch.randn(n, cols + pad, generator=g, device="cuda")[:, :cols]


# (tokens, width, k, r, outputs, columns of padding): remainders of the 32, 64 and 128 tiles and of 16-row steps,
# one step only, products that fill the chip and products that leave it idle (which tile and how many pieces of K
# each takes is the dispatch's choice; every pair is forced in test_gpu_debug_bounds.py)
@pytest.mark.parametrize("N,d,k,r,d_out,pad", [
    (1, 5, 2, 2, 1, 0), (33, 31, 3, 0, 65, 1), (130, 129, 8, 9, 127, 3), (2048, 512, 16, 16, 512, 0),
    (2049, 257, 40, 24, 511, 2), (8191, 1023, 64, 63, 1000, 1), (8192, 1024, 64, 64, 1024, 0), (700, 1024, 128, 128, 4096, 4),
])
def test_products_of_fp32_storage(N, d, k, r, d_out, pad):
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    X, dY = _rows(N, d, pad, g), _rows(N, d_out, pad, g)
    W = _rows(d_out, d, pad, g)
    P = torch.linalg.qr(torch.randn(d, k + r, generator=g, device="cuda", dtype=torch.float64))[0].float()
    b = api.Basis(d, k, r, torch.float32)
    c = 1.75
    b.set(P[:, :k].contiguous(), P[:, k:].contiguous(), c)
    Z = b.compress(X)
    _close(Z, X.double() @ P.double(), d, "compress")
    Y, Z2 = b.linear_forward(X, W)
    _close(Y, X.double() @ W.double().t(), d, "forward")
    assert torch.equal(Z2, Z)
    _close(b.reconstruct(Z), torch.cat([Z[:, :k], c * Z[:, k:]], 1).double() @ P.double().t(), k + r, "reconstruct")
    M = dY.double().t() @ Z.double()
    M[:, k:] *= c
    want = M @ P.double().t()
    wide = torch.zeros(d_out, d + pad, device="cuda")
    dW = b.weight_grad(dY, Z, out=wide[:, :d])
    # (two products in a row; the inner one is rounded to fp32)
    _close(dW, want, 2 * (N + k + r), "weight gradient")
    first = dW.clone()
    b.weight_grad(dY, Z, out=dW, accumulate=True)
    _close(dW, 2 * first.double(), N + k + r, "accumulated weight gradient")
    assert not wide[:, d:].any()
    C = b.gram(X)
    assert torch.equal(C, C.t())
    _close(C, X.double().t() @ X.double(), 2 * N, "gram")   # (same-signed diagonal sums add up faster than random ones)
    assert torch.equal(b.compress(X), Z) and torch.equal(b.weight_grad(dY, Z), first)
