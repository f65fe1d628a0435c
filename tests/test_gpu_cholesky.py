"""The factorisation inside Cholesky-QR at the sizes where its kernel changes: blocks of 32 columns (one block, a last
block of one column or one short), clusters above the portable eight CTAs, the kernel for more than 512 columns, and a
panel whose rank ends inside a block.  Through prac_draw_random without a principal part, which orthonormalises a
Gaussian block: its thin QR factor with positive diagonal is unique.

Bounds: each column of Q to 1e-4 (fp32 panel; that R is exact to double is checked on ill-conditioned panels), and the orthonormality that rounding Q to fp32 leaves,
||Q^T Q - I||_F of about n 2^-24 with a constant of order one (8.5e-6 measured at 512 columns)."""
import numpy as np
import pytest
import torch

from oracle import prac_oracle as orc
from paper_2602_23111_b200 import inputs

pytestmark = pytest.mark.gpu


def f64(t):
    return t.detach().to(torch.float32).cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("r", [1, 8, 31, 32, 33, 65, 256, 257, 320, 511, 512, 513, 640])
def test_random_basis_is_the_unique_qr_factor(r):
    from paper_2602_23111_b200 import api
    d = max(256, 2 * r + 19)
    b = api.Basis(d, 0, r, torch.float32)
    b.draw_random(seed=11, draw_counter=5)
    assert b.status() == api.PRAC_OK
    Q = f64(b.projection()[0])
    Q0 = orc.random_basis(np.zeros((d, 0)), orc.gaussian_draw(11, 5, d, r))
    assert np.max(np.linalg.norm(Q - Q0, axis=0)) <= 1e-4
    assert np.linalg.norm(Q.T @ Q - np.eye(r)) <= max(1e-5, 2e-5 * r / 512)
    b.draw_random(seed=11, draw_counter=5)
    assert np.array_equal(f64(b.projection()[0]), Q)          # sums in a fixed order, whoever is first


@pytest.mark.parametrize("r", [1, 8, 31, 32, 33, 64, 65, 97, 257, 320, 512])
def test_cooperative_kernel_serves_where_no_cluster_can_be_placed(r):
    # whether the cluster fits is asked for every launch: where it does not, the kernel for more than 512 columns takes over
    from paper_2602_23111_b200 import api
    d = max(256, 2 * r + 19)
    b = api.Basis(d, 0, r, torch.float32)
    api.lib.prac_debug_force_cooperative_cholesky(1)
    try:
        b.draw_random(seed=11, draw_counter=5)
        Q = f64(b.projection()[0])
        b.draw_random(seed=11, draw_counter=5)
        assert b.status() == api.PRAC_OK
    finally:
        api.lib.prac_debug_force_cooperative_cholesky(0)
    assert np.array_equal(f64(b.projection()[0]), Q)
    Q0 = orc.random_basis(np.zeros((d, 0)), orc.gaussian_draw(11, 5, d, r))
    assert np.max(np.linalg.norm(Q - Q0, axis=0)) <= 1e-4
    assert np.linalg.norm(Q.T @ Q - np.eye(r)) <= max(1e-5, 2e-5 * r / 512)


@pytest.mark.parametrize("k, rank", [(256, 100), (128, 33), (64, 64)])
def test_panel_whose_rank_ends_inside_a_block(k, rank):
    # pivots are replaced from column `rank` on, in every block after it; the extra pass makes the rest orthonormal
    from paper_2602_23111_b200 import api
    N, d = 700, 640
    X = inputs.make_planted(N, d, rank, seed=31, dtype="f32", exact_rank=True)
    b = api.Basis(d, k, 8, torch.float32)
    b.fit(X.cuda(), seed=6)
    assert b.status() == api.PRAC_OK
    U, X64 = f64(b.get()[0]), f64(X)
    assert np.linalg.norm(U.T @ U - np.eye(k)) <= 1e-5
    assert np.linalg.norm(X64 - X64 @ U @ U.T) <= 1e-4 * np.linalg.norm(X64)


@pytest.mark.parametrize("cooperative", [0, 1])
@pytest.mark.parametrize("n", [32, 33, 256, 257, 512, 513])
@pytest.mark.parametrize("kappa", [1e2, 1e5, 1e6])
def test_inverse_factor_of_an_ill_conditioned_panel_is_exact_to_double(n, kappa, cooperative):
    # Singular values from 1 to 1 / kappa, columns mixed.  The panel's last n rows are eps I, so that those rows of Q are eps
    # R^-1, element by element to fp32 (2^-22).  Rounding V^T V and its factor to double turns R^-1 by about kappa^2 2^-53
    # (a tenth of it measured, at all sizes); a step in fp32, or with ten bits of a double lost, is far beyond that at 1e5 and 1e6.
    # Pivots stay above 1e-13 of their column's norm, so none is replaced.
    from paper_2602_23111_b200 import api
    d = n + 300 + n // 2
    rng = np.random.default_rng(n)
    A = np.linalg.qr(rng.standard_normal((d - n, n)))[0] * np.logspace(0, -np.log10(kappa), n)
    A = A @ np.linalg.qr(rng.standard_normal((n, n)))[0]
    eps = 2.0 ** -10 / kappa
    V = np.concatenate([A, eps * np.eye(n)]).astype(np.float32)
    R = np.linalg.qr(V.astype(np.float64), mode="r")
    R *= np.sign(np.diag(R))[:, None]
    exact = np.linalg.solve(R, np.eye(n))
    Vd, word = torch.from_numpy(V).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    Q = torch.empty_like(Vd)
    ws = torch.empty(api.lib.prac_debug_cholqr_ws_bytes(d, n), dtype=torch.uint8, device="cuda")
    api.lib.prac_debug_force_cooperative_cholesky(cooperative)
    try:
        st = api.lib.prac_debug_cholqr(Vd.data_ptr(), Q.data_ptr(), d, n, ws.data_ptr(), ws.numel(), word.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
    finally:
        api.lib.prac_debug_force_cooperative_cholesky(0)
    assert st == api.PRAC_OK and int(word.item()) == 0
    got = f64(Q)[-n:] / eps
    off = np.linalg.norm(got - exact) / np.linalg.norm(exact)
    assert off <= 2.0 ** -22 + 2.0 ** -53 * kappa ** 2


def test_quotients_of_the_elimination_against_division():
    # One step of the cubic iteration leaves 2^-60, its three roundings 2^-53 each with factors of one at most: two units of the
    # last place, 2^-52 relative, of the correctly rounded quotient.  Pivots: squared norms of fp32 columns.
    import ctypes
    from paper_2602_23111_b200 import api
    n = 1 << 20
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    mantissa = 1 + torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    mantissa[:64] = 1 + torch.arange(64, device="cuda", dtype=torch.float64) * 2.0 ** -52
    mantissa[64:128] = 2 - torch.arange(1, 65, device="cuda", dtype=torch.float64) * 2.0 ** -52
    exponent = torch.randint(-300, 280, (n,), generator=g, device="cuda")
    b = torch.ldexp(mantissa, exponent)
    a = torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * torch.ldexp(torch.ones_like(b), exponent)
    q = torch.empty_like(a)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    assert api.lib.prac_debug_quotients(p(a), p(b), p(q), n, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == api.PRAC_OK
    exact = a / b
    assert float(((q - exact) / exact).abs().max()) <= 2 * 2.0 ** -52
