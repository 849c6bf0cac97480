"""Zero columns of the operand tables of the low-rank term: by the quads' own threads, or as items of their own (ranks 4
and 8, rows of several slots).  The tables lie in scratch that an earlier call of a higher rank has filled, so a zero that
is not written shows in the outputs.  A projection at an address that is not a multiple of 16 takes the kernel that writes
whole 16-byte chunks: the same tables, and so the same bits."""
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


@pytest.mark.parametrize("own", [None, False, True])          # one layer; gate and up; each with its own projection
@pytest.mark.parametrize("r", [4, 8, 12, 16, 24, 64])
@pytest.mark.parametrize("T,nb,d_out", [(256, 2, 136), (130, 2, 136), (100, 3, 136), (16, 17, 136),   # 1, 2, 3, 17 slots
                                        (16, 17, 4408)])         # enough columns for rank 8's own threads
def test_operand_zeros(ctx, T, nb, d_out, r, own):
    d_in, seed, rows = 128, 3, nb * T
    pts = [(0.5, 7), (-0.5, 7)] if nb == 2 else [(0.25 * (1 + j) / nb, j) for j in range(nb)]
    X = normal((rows, d_in), 1, DEV, dtype=torch.bfloat16)
    W = [normal((d_out, d_in), 2 + i, DEV, std=d_in ** -0.5, dtype=torch.bfloat16) for i in range(2)]
    U = [normal((d_in, 96), 4 + i, DEV, std=d_in ** -0.5) for i in range(2)]
    C = [normal((d_out, 96), 6 + i, DEV, std=0.3) for i in range(2)]
    Y = torch.empty(rows, d_out, dtype=torch.bfloat16, device=DEV)

    def run(rank, shift):
        Ur, Cr = [u[:, :rank].contiguous() for u in U], [c[:, :rank].contiguous() for c in C]
        L = [zo.make_layer(W[i], Ur[i] if own else Ur[0], Cr[i], i) for i in range(2)]
        P = []
        for u in Ur:
            buf = torch.empty(rows * rank + 1, device=DEV)
            p = buf[shift:shift + rows * rank].view(rows, rank)
            q = torch.empty(rows, rank, device=DEV)
            zo.zoact_lowrank_proj(ctx, X, u, q)
            p.copy_(q)
            P.append(p)
        if own is None:
            zo.zoact_multi_forward(ctx, L[0], X, T, False, pts, seed, Y, P=P[0])
        else:
            zo.zoact_multi_forward_gated(ctx, L[0], L[1], X, T, False, pts, seed, Y, P_gate=P[0],
                                         P_up=P[1] if own else P[0])
        torch.cuda.synchronize()
        assert ctx.device_status() == 0
        return Y.clone()

    run(96, 0)                               # every column of the tables' scratch is taken
    aligned = run(r, 0)
    run(96, 0)
    assert torch.equal(aligned, run(r, 1))
    n64 = lambda t: t.double().cpu().numpy()
    out = []
    for i in range(1 if own is None else 2):
        x, w, u, c = n64(X), n64(W[i]), n64(U[i if own else 0][:, :r]), n64(C[i][:, :r])
        blk = []
        for b, (e, q) in enumerate(pts):
            xb = x[b * T:(b + 1) * T]
            blk.append(xb @ w.T + (xb @ u) @ (c + e * philox.perturbation(seed, i, q, d_out, r)).T)
        out.append(np.concatenate(blk))
    ref = out[0] if own is None else layers.silu(out[0]) * out[1]
    # half an ulp of bf16, and 2^-14 of terms of order one for the two-part operands
    assert np.all(np.abs(n64(aligned) - ref) <= 2.0 ** -8 * np.abs(ref) + 2e-3)
