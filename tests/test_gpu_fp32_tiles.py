"""fp32 projection and pair forward at the edges of their tiles, against the fp64 oracle.

Bounds per element: a chain of d_in fp32 FMAs errs by at most d_in 2^-24 sum |terms|; 4 sqrt(d_in) of that, as the other
fp32 tests use, plus the same of the low-rank term.
"""
import numpy as np
import pytest
import torch

import paper_2607_01125_gb300 as zo
from oracle import layers, philox
from synth import normal

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    c = zo.Context(0)
    yield c
    assert c.device_status() == 0
    c.close()


@pytest.mark.parametrize("rows,d_in,r", [(1, 4, 1), (37, 100, 9), (64, 256, 8), (2500, 1024, 33), (130, 1028, 5)])
def test_projection_fp32(ctx, rows, d_in, r):
    X, U = normal((rows, d_in), 1, DEV), normal((d_in, r), 2, DEV)
    P = torch.empty(rows, r, device=DEV)
    zo.zoact_lowrank_proj(ctx, X, U, P)
    torch.cuda.synchronize()
    Xn, Un = X.double().cpu().numpy(), U.double().cpu().numpy()
    bound = 4 * np.sqrt(d_in) * 2.0 ** -24 * (np.abs(Xn) @ np.abs(Un))
    assert np.all(np.abs(P.double().cpu().numpy() - Xn @ Un) <= bound)


@pytest.mark.parametrize("d_in,d_out,T,r,shared,nb", [
    (4, 8, 1, 1, False, 2),              # one output tile of 16, one K chunk
    (300, 72, 23, 6, True, 2),           # ragged everything; more chunks than stages
    (256, 256, 250, 8, False, 2),        # 32 x 32 tiles
    (128, 520, 700, 36, False, 3),       # 64 x 64 tiles straddling blocks, two table passes
    (512, 1032, 300, 4, True, 9),        # 64 x 64 tiles, nine blocks of one input
])
def test_pair_forward_fp32_tiles(ctx, d_in, d_out, T, r, shared, nb):
    seed, lid = 5, 2
    pts = [(0.5, 3), (-0.5, 3)] if nb == 2 else [(0.0, 0)] + [(0.25 * (j + 1) / nb, j) for j in range(nb - 1)]
    X = normal(((T if shared else nb * T), d_in), 1, DEV)
    W, U = normal((d_out, d_in), 2, DEV, std=d_in ** -0.5), normal((d_in, r), 3, DEV, std=d_in ** -0.5)
    C = normal((d_out * r,), 4, DEV, std=0.3)
    Y = torch.full((nb * T, d_out), float("nan"), device=DEV)
    zo.zoact_multi_forward(ctx, zo.make_layer(W, U, C, lid), X, T, shared, pts, seed, Y, act=zo.ACT_RELU)
    torch.cuda.synchronize()
    n64 = lambda t: t.double().cpu().numpy()
    Xn, Wn, Un, Cn = n64(X), n64(W), n64(U), n64(C).reshape(d_out, r)
    for b, (c, q) in enumerate(pts):
        x = Xn if shared else Xn[b * T:(b + 1) * T]
        Tb = Cn + c * philox.perturbation(seed, lid, q, d_out, r)
        ref = np.maximum(x @ Wn.T + (x @ Un) @ Tb.T, 0)
        lr = np.abs(x) @ np.abs(Un) @ np.abs(Tb).T
        bound = 4 * np.sqrt(d_in) * 2.0 ** -24 * (np.abs(x) @ np.abs(Wn).T + lr) + 1e-6 * lr + 1e-7
        assert np.all(np.abs(n64(Y[b * T:(b + 1) * T]) - ref) <= bound), b


def _check_projection(X, U, P):
    Xn, Un = X.double().cpu().numpy(), U.double().cpu().numpy()
    bound = 4 * np.sqrt(X.shape[1]) * 2.0 ** -24 * (np.abs(Xn) @ np.abs(Un))
    assert np.all(np.abs(P.double().cpu().numpy() - Xn @ Un) <= bound)


@pytest.mark.parametrize("rows,d_in,r", [(9001, 1024, 40), (16384, 64, 96), (4097, 512, 72),   # blocks: many rows, ranks
                                         (700, 64, 24), (1000, 1024, 36), (305, 1024, 64)])     # four rows a warp
def test_projection_fp32_forms(ctx, rows, d_in, r):
    X, U = normal((rows, d_in), 1, DEV), normal((d_in, r), 2, DEV)
    P = torch.full((rows, r), float("nan"), device=DEV)
    zo.zoact_lowrank_proj(ctx, X, U, P)
    torch.cuda.synchronize()
    _check_projection(X, U, P)


def test_projection_fp32_first_call_captured():
    # K-splits in scratch that a capture cannot allocate: the form without scratch
    X, U = normal((4096, 1024), 1, DEV), normal((1024, 64), 2, DEV)
    P = torch.full((4096, 64), float("nan"), device=DEV)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        c = zo.Context(0)
        c.sync_stream()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            zo.zoact_lowrank_proj(c, X, U, P)
        g.replay()
        torch.cuda.synchronize()
    _check_projection(X, U, P)
    c.close()
