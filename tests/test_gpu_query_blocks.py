"""Several evaluation blocks on a shared input with 16-bit outputs on CTA pairs: the low-rank term of each block goes on
the epilogue warps' matrix instruction from Z tables in operand order.  Sizes at the edges of the layout: ranks around
the groups of eight (and ones that split a Philox group), columns that end inside a pass, rows that end inside a warp's
32 and a CTA without rows, zero and repeated evaluation points."""
import numpy as np
import pytest
import torch

import paper_2607_01125_gb300 as zo
from oracle import layers
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
