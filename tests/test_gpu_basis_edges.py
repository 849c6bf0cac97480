"""The one-shot basis at the edges of its kernels' ranges, against the same subspace iteration in fp64.

Singular values fall as 0.93^i (columns well apart), so every column is determined: its error is fp32's (2^-24) times the
condition of its eigenvector, 1 / (1 - 0.93^2) = 7.4 relative to its own eigenvalue times sigma_1^2 / sigma_i^2 for the
Gram matrix's rounding -- at column 8, 3e-7 x 7.4 x 2.9 < 1e-5; 1e-4 is asserted for columns up to 8.
"""
import numpy as np
import pytest
import torch

import paper_2607_01125_gb300 as zo
from oracle import basis

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    c = zo.Context(0)
    yield c
    assert c.device_status() == 0
    c.close()


def _tokens(n, d, rank, dtype, seed, scale=1.0, decay=0.93):
    g = torch.Generator(device=DEV).manual_seed(seed)
    B = torch.linalg.qr(torch.randn(d, rank, generator=g, device=DEV))[0].T
    A = torch.linalg.qr(torch.randn(max(n, rank), rank, generator=g, device=DEV))[0][:n]
    s = decay ** torch.arange(rank, device=DEV, dtype=torch.float32)
    return ((A * s) @ B * scale * (n * d) ** 0.5 / 4).to(dtype)


@pytest.mark.parametrize("n,d,r,over,dtype", [
    (40, 16, 1, 0, torch.bfloat16),          # k = 1
    (100, 64, 1, 1, torch.float16),          # k = 2
    (100, 72, 2, 1, torch.bfloat16),         # k = 3 (odd: the schedule's dummy)
    (333, 1000, 17, 16, torch.bfloat16),     # k = 33, ragged tokens and columns
    (512, 520, 48, 16, torch.float16),       # k = 64: the last of the shared-memory kernels
    (512, 520, 49, 16, torch.bfloat16),      # k = 65: the first of the chip-wide ones
    (700, 648, 100, 29, torch.float16),      # k = 129: odd, five panels
    (1200, 640, 256, 256, torch.bfloat16),   # k = 512: the largest
    (40, 400, 8, 60, torch.bfloat16),        # fewer tokens than columns sought: Cholesky with a shift
    (3000, 128, 8, 16, torch.float16),       # many more tokens than columns
    (300, 128, 8, 70, torch.float32),        # fp32 tokens, k = 78
])
def test_basis_edges(ctx, n, d, r, over, dtype):
    X = _tokens(n, d, min(n, d), dtype, n + d)
    k = r + over
    U = torch.empty(d, r, device=DEV)
    ev = torch.empty(k, device=DEV)
    zo.zoact_basis_init(ctx, X, r, U, oversample=over, n_iter=8, seed=9, evals_out=ev)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    Un = U.double().cpu().numpy()
    np.testing.assert_allclose(Un.T @ Un, np.eye(r), atol=1e-5)
    ref, theta = basis.subspace_iteration(basis.gram(X.double().cpu().numpy()), r, over, 8, 9)
    top = min(r, 8)
    np.testing.assert_allclose(Un[:, :top], ref[:, :top], atol=1e-4)
    np.testing.assert_allclose(ev.cpu().numpy()[:top], np.asarray(theta)[:top], rtol=1e-4)


@pytest.mark.parametrize("scale", [1e-4, 1.0, 1e3])
def test_basis_fp16_scales(ctx, scale):
    # fp16 tokens far from unit scale: the three-term factors must keep their small parts
    X = _tokens(512, 512, 128, torch.float16, 3, scale)
    U = torch.empty(512, 8, device=DEV)
    zo.zoact_basis_init(ctx, X, 8, U, oversample=16, n_iter=8, seed=2)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0 and bool(torch.isfinite(X).all())
    ref, _ = basis.subspace_iteration(basis.gram(X.double().cpu().numpy()), 8, 16, 8, 2)
    np.testing.assert_allclose(U.double().cpu().numpy(), ref, atol=1e-4)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("n,d,r,over", [(300, 256, 8, 16),       # k = 24
                                        (300, 256, 1, 0),        # k = 1
                                        (300, 256, 64, 15),      # k = 79: chip-wide
                                        (2100, 256, 8, 33)])     # a Gram matrix in every type, k = 41
def test_basis_nonfinite_tokens(ctx, n, d, r, over, dtype, bad):
    # one bad element: no finite entry in any column, the status says so, and the context stays usable
    X = _tokens(n, d, 128, dtype, 5)
    X[7, 11] = bad
    U = torch.zeros(d, r, device=DEV)
    ev = torch.zeros(r + over, device=DEV)
    zo.zoact_basis_init(ctx, X, r, U, oversample=over, n_iter=2, seed=3, evals_out=ev)
    torch.cuda.synchronize()
    assert ctx.device_status() == -4
    assert not bool(torch.isfinite(U).any())
    X[7, 11] = 0.0
    zo.zoact_basis_init(ctx, X, r, U, oversample=over, n_iter=2, seed=3, evals_out=ev)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0 and bool(torch.isfinite(U).all()) and bool(torch.isfinite(ev).all())


def test_basis_fast_falling_fp32(ctx):
    # k = 78 columns of a spectrum that is spent after ~12: Q^T (G Q) is not positive within fp32's rounding.  Column i errs
    # by 2^-24 times its eigenvalue's distance: at i = 3, 3e-7 x 1.33 x (sigma_1 / sigma_4)^2 = 64, 3e-5
    X = _tokens(300, 128, 128, torch.float32, 8, decay=0.5)
    U, ev = torch.empty(128, 8, device=DEV), torch.empty(78, device=DEV)
    zo.zoact_basis_init(ctx, X, 8, U, oversample=70, n_iter=8, seed=9, evals_out=ev)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    Un = U.double().cpu().numpy()
    np.testing.assert_allclose(Un.T @ Un, np.eye(8), atol=1e-5)
    ref, theta = basis.subspace_iteration(basis.gram(X.double().cpu().numpy()), 8, 70, 8, 9)
    np.testing.assert_allclose(Un[:, :4], ref[:, :4], atol=1e-4)
    np.testing.assert_allclose(ev.cpu().numpy()[:4], np.asarray(theta)[:4], rtol=1e-4)


def test_basis_indefinite_gram(ctx):
    # Rank one and many fp32 tokens: the Gram matrix's chains leave eigenvalues down to -7e-6 of its trace (a model of the
    # chains in numpy), and the Ritz problem of the k = 78 largest in absolute value is indefinite.  An entry of G errs by
    # sqrt(n) 2^-24 = 4e-5 of itself (a random walk), the eigenvector by 2 / sqrt(d) of that.
    n, d, r, over = 400_000, 128, 8, 70
    g = torch.Generator(device=DEV).manual_seed(4)
    a = torch.rand(d, generator=g, device=DEV) + 0.5
    X = (torch.rand(n, 1, generator=g, device=DEV) + 0.5) * a
    U, ev = torch.empty(d, r, device=DEV), torch.empty(r + over, device=DEV)
    zo.zoact_basis_init(ctx, X, r, U, oversample=over, n_iter=8, seed=9, evals_out=ev)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    ev = ev.double().cpu().numpy()
    assert np.all(np.diff(ev) <= 0) and ev[-1] < 0
    np.testing.assert_allclose(ev[0], float((X.double() ** 2).sum()), rtol=1e-3)
    Un = U.double().cpu().numpy()
    np.testing.assert_allclose(Un.T @ Un, np.eye(r), atol=1e-5)
    an = a.double().cpu().numpy()
    np.testing.assert_allclose(Un[:, 0], an / np.linalg.norm(an), atol=1e-4)
