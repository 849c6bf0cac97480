"""Several evaluation blocks on a shared input with 16-bit outputs on CTA pairs: the low-rank term of each block goes on
the epilogue warps' matrix instruction from Z tables in operand order.  Sizes at the edges of the layout: ranks around
the groups of eight (and ones that split a Philox group), columns that end inside a pass, rows that end inside a warp's
32 and a CTA without rows, zero and repeated evaluation points.  And the losses of several blocks."""
import numpy as np
import pytest
import torch

import paper_2607_01125_gb300 as zo
from oracle import layers, loss as oloss
from test_gpu_multi import DEV, _oracle, ctx, normal, np64  # noqa: F401  (ctx: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gated", [False, True])
@pytest.mark.parametrize("T,d_out,r,dt", [(257, 264, 1, torch.bfloat16), (300, 328, 6, torch.float16),
                                          (353, 72, 8, torch.bfloat16), (289, 200, 9, torch.bfloat16),
                                          (512, 136, 16, torch.float16), (257, 296, 17, torch.bfloat16),
                                          (400, 168, 24, torch.bfloat16), (320, 520, 32, torch.float16)])
def test_query_blocks_edges(ctx, gated, T, d_out, r, dt):  # noqa: F811
    d_in, seed = 256, 5
    pts = [(0.0, 1), (0.25, 1), (-0.125, 2), (0.0, 3), (0.25, 2)]
    X = normal((T, d_in), 51, DEV, dtype=dt)
    Wg = normal((d_out, d_in), 52, DEV, std=d_in ** -0.5, dtype=dt)
    Wu = normal((d_out, d_in), 53, DEV, std=d_in ** -0.5, dtype=dt)
    U = normal((d_in, r), 54, DEV) / np.sqrt(d_in)
    Cg, Cu = normal((d_out * r,), 56, DEV, std=0.2), normal((d_out * r,), 57, DEV, std=0.2)
    n = len(pts) * T
    Y = torch.full((n + 8, d_out), 7.0, dtype=dt, device=DEV)
    g, _, _ = _oracle(np64(Wg), np64(U), np64(Cg).reshape(d_out, r), np64(X), pts, T, True, seed, 0)
    if gated:
        zo.zoact_multi_forward_gated(ctx, zo.make_layer(Wg, U, Cg, 0), zo.make_layer(Wu, U, Cu, 1), X, T, True, pts,
                                     seed, Y[:n])
        u, _, _ = _oracle(np64(Wu), np64(U), np64(Cu).reshape(d_out, r), np64(X), pts, T, True, seed, 1)
        ref = layers.silu(g) * u
    else:
        zo.zoact_multi_forward(ctx, zo.make_layer(Wg, U, Cg, 0), X, T, True, pts, seed, Y[:n])
        ref = g
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    # half an ulp of the stored type, and the operands of C p held to 2^-16 (products of d_in and r terms of order one)
    rel = {torch.bfloat16: 2.0 ** -8, torch.float16: 2.0 ** -11}[dt]
    err = np.abs(np64(Y[:n]) - ref)
    assert np.all(err <= rel * np.abs(ref) + 2e-4 * np.abs(ref).max()), err.max()
    assert torch.all(Y[n:] == 7.0)
    # equal points give equal bits
    b = Y[:n].view(len(pts), T, d_out)
    assert torch.equal(b[0], b[3])


@pytest.mark.parametrize("T,n,nb,dt,with_target", [(640, 1000, 7, torch.float32, False), (640, 1000, 6, torch.float32, True),
                                                   (641, 1000, 10, torch.bfloat16, True), (1, 8, 2, torch.float16, True),
                                                   (1, 1, 17, torch.float32, True), (997, 643, 9, torch.float16, False)])
def test_loss_blocks_edges(ctx, T, n, nb, dt, with_target):  # noqa: F811
    # a vector more than the grid's threads, blocks past a round of four, the scalar path, one element
    y0 = normal((T, n), 61, DEV)
    Y = torch.cat([y0] + [y0 + 1e-2 * normal((T, n), 62 + j, DEV) for j in range(nb - 1)]).to(dt)
    tgt = normal((T, n), 80, DEV, dtype=dt) if with_target else None
    out = torch.full((2 * nb,), 7.0, dtype=torch.float64, device=DEV)
    mu = 1e-3
    for _ in range(2):                       # the ticket is back at zero
        zo.zoact_loss_multi(ctx, Y, T, nb, mu, out, target=tgt)
    torch.cuda.synchronize()
    o, Yn = out.cpu().numpy(), np64(Y)
    L, a = oloss.loss_queries(Yn, T, nb, None if tgt is None else np64(tgt), mu)
    # fp32 differences, squares and sums of 8 a vector (10 roundings), then compensated sums
    np.testing.assert_allclose(o[:nb], L, rtol=16 * 2.0 ** -24)
    t = 0.0 if tgt is None else np64(tgt)
    for j in range(1, nb):
        scale = np.mean(np.abs((Yn[j * T:(j + 1) * T] - Yn[:T]) * (Yn[j * T:(j + 1) * T] + Yn[:T] - 2 * t))) / mu
        assert abs(o[nb + j - 1] - a[j - 1]) <= 16 * 2.0 ** -24 * scale + 2.0 ** -50 * abs(a[j - 1])
    assert o[-1] == 7.0


@pytest.mark.parametrize("T,n,nb,dt,with_target", [
    (1027, 1000, 5, torch.bfloat16, True),    # one round of four blocks and a last thread group of one vector
    (1027, 1000, 6, torch.float16, False),    # a block past it
    (1027, 1000, 9, torch.bfloat16, False),   # two rounds
    (2055, 1000, 2, torch.bfloat16, True),    # one block beside y0
    (2055, 1000, 2, torch.float32, False),
    (5603, 1000, 2, torch.bfloat16, True),    # ... with two CTAs per SM
    (5603, 1000, 2, torch.float32, False),
])
def test_loss_blocks_rounds(ctx, T, n, nb, dt, with_target):  # noqa: F811
    test_loss_blocks_edges(ctx, T, n, nb, dt, with_target)


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("nb", [2, 3])
def test_loss_blocks_large_values(ctx, nb, dt):  # noqa: F811
    # a thread's sum of squares fits fp32 (8 or 16 values of 2e18 a vector group), sixteen threads' do not
    T, n, mu = 640, 1000, 1.0
    Y = (2e18 * (1.0 + 0.25 * torch.rand(nb * T, n, device=DEV))).to(dt)
    out = torch.zeros(2 * nb, dtype=torch.float64, device=DEV)
    zo.zoact_loss_multi(ctx, Y, T, nb, mu, out)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    o, Yn = out.cpu().numpy(), np64(Y)
    L, a = oloss.loss_queries(Yn, T, nb, None, mu)
    np.testing.assert_allclose(o[:nb], L, rtol=16 * 2.0 ** -24)
    for j in range(1, nb):
        scale = np.mean(np.abs((Yn[j * T:(j + 1) * T] - Yn[:T]) * (Yn[j * T:(j + 1) * T] + Yn[:T])))
        assert abs(o[nb + j - 1] - a[j - 1]) <= 16 * 2.0 ** -24 * scale
