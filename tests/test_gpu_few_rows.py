"""The pair forward of fewer than 256 rows of X: the few-row kernel at the edges of its tiles, and the kernel that is
chosen by the estimated times, against the fp64 oracle.

Tolerances, per element: fp32 accumulation 8 sqrt(d_in) 2^-24 sum |terms| (the K ranges of a cluster are added in a
fixed order, so the bound of one sum holds), INT4 weights rounded once to bf16 (2^-9 of sum |x w|); the other route's
two-part operands of the low-rank term (2^-14 of its |terms|; the few-row kernel has three parts).  Gated outputs: the
same bound on gate and up, through |d silu| <= 1.1, plus the approximate exponential and reciprocal in SiLU (2^-20 of the
product).
"""
import numpy as np
import pytest
import torch

import paper_2607_01125_gb300 as zo
from oracle import layers, philox
from synth import normal, quantize_int4_g128

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    c = zo.Context(0)
    yield c
    assert c.device_status() == 0
    c.close()


@pytest.fixture(params=["few", "chosen"], autouse=True)
def route(request, monkeypatch):
    if request.param == "few":
        monkeypatch.setenv("ZOACT_PAIR_KERNEL", "few")
    return request.param


def np64(t):
    return t.detach().double().cpu().numpy()


def _layer(d_in, d_out, r, wtype, seed, lid, U=None):
    U = normal((d_in, r), seed + 1, DEV) / np.sqrt(d_in) if U is None else U
    C = normal((d_out * r,), seed + 2, DEV, std=0.3)
    Wf = normal((d_out, d_in), seed, DEV, std=0.02)
    if wtype == "int4":
        packed, scales = quantize_int4_g128(Wf)
        L = zo.make_layer(packed, U, C, lid, w_scales=scales, wtype=zo.DT_INT4_G128, d_in=d_in)
        return L, layers.dequant_int4_g128(packed.cpu().numpy(), scales.float().cpu().numpy(), d_in), U, C
    W = Wf.to({"bf16": torch.bfloat16, "fp16": torch.float16}[wtype])
    return zo.make_layer(W, U, C, lid), np64(W), U, C


def _ref(W, U, C, X, T, shared, pts, seed, lid, r, int4, split):
    """Blocks of outputs and the bound of their error."""
    Xn, Un, Cn = np64(X), np64(U), np64(C).reshape(W.shape[0], r)
    out, bound = [], []
    for b, (c, q) in enumerate(pts):
        x = Xn if shared else Xn[b * T:(b + 1) * T]
        Tb = Cn + c * philox.perturbation(seed, lid, q, W.shape[0], r)
        out.append(x @ W.T + (x @ Un) @ Tb.T)
        base = np.abs(x) @ np.abs(W).T
        lr = np.abs(x @ Un) @ np.abs(Tb).T + (np.abs(x) @ np.abs(Un)) @ np.abs(Tb).T * 2.0 ** -10
        bound.append(8 * np.sqrt(W.shape[1]) * 2.0 ** -24 * (base + lr) + (2.0 ** -14 * lr if split else 0.0) +
                     (2.0 ** -9 * base if int4 else 0.0) + 1e-6)
    return np.concatenate(out), np.concatenate(bound)


@pytest.mark.parametrize("wtype,d_in,d_out,T,r,shared,nb,gated", [
    ("bf16", 64, 8, 1, 1, False, 2, False),         # one K-block, two rows, eight outputs
    ("bf16", 1000, 520, 37, 5, False, 2, False),    # ragged K and N tiles, rank 5
    ("bf16", 4096, 1024, 16, 16, False, 2, False),  # eight K ranges; 32 rows
    ("fp16", 1792, 5120, 33, 16, False, 2, False),  # six: seven would fill the CTA slots, but not as clusters at once
    ("fp16", 2048, 136, 127, 32, False, 2, False),  # 254 rows
    ("bf16", 8200, 256, 17, 16, True, 2, False),    # shared input, K ending inside a block
    ("fp16", 512, 264, 255, 8, True, 2, False),     # the most rows
    ("bf16", 512, 384, 14, 16, False, 17, False),   # 17 blocks of 14 rows
    ("bf16", 1024, 200, 9, 32, True, 5, True),      # gated, shared, five blocks
    ("bf16", 4096, 640, 100, 16, False, 2, True),   # gated, 200 rows: one CTA per SM, rows in several chunks
    ("bf16", 4096, 256, 64, 32, False, 2, True),
    ("bf16", 512, 264, 60, 40, False, 2, False),    # rank above 32: extra K-blocks
    ("fp16", 576, 264, 21, 70, False, 3, True),
    ("int4", 128, 8, 1, 4, False, 2, False),        # one scale group
    ("int4", 14336, 512, 64, 32, False, 2, False),  # eight K ranges, odd ones starting inside a scale group
    ("int4", 1152, 264, 100, 16, False, 2, False),  # 9 groups; 200 rows
    ("int4", 2048, 136, 255, 3, True, 2, False),
    ("int4", 1024, 200, 40, 16, False, 2, True),
    ("int4", 1024, 520, 120, 32, True, 3, True),    # gated, rank 32: one CTA per SM
])
def test_few_rows(ctx, route, wtype, d_in, d_out, T, r, shared, nb, gated):
    seed, eps = 11, 0.5
    pts = [(eps, 7), (-eps, 7)] if nb == 2 else [(0.0, 0)] + [(eps * (1 + j) / nb, j) for j in range(nb - 1)]
    L, W, U, C = _layer(d_in, d_out, r, wtype, 100, 3)
    dt = torch.float16 if wtype == "fp16" else torch.bfloat16
    X = normal(((T if shared else nb * T), d_in), 5, DEV, dtype=dt)
    L2, W2, U2, C2 = _layer(d_in, d_out, r, wtype, 200, 4)      # gated: its own basis, a second projection

    def reference(split):
        ref, bound = _ref(W, U, C, X, T, shared, pts, seed, 3, r, wtype == "int4", split)
        if not gated:
            return ref, bound
        u, ub = _ref(W2, U2, C2, X, T, shared, pts, seed, 4, r, wtype == "int4", split)
        g = layers.silu(ref)
        return g * u, 1.1 * bound * np.abs(u) + np.abs(g) * ub + 1.1 * bound * ub + 2.0 ** -20 * np.abs(g * u)

    for ydt in (torch.float32, dt):
        ref, bound = reference(route == "chosen" and ydt != torch.float32)   # (fp32 outputs keep the few-row kernel)
        outs = []
        for _ in range(2):
            Y = torch.full((nb * T, d_out), float("nan"), dtype=ydt, device=DEV)
            if gated:
                zo.zoact_multi_forward_gated(ctx, L, L2, X, T, shared, pts, seed, Y)
            else:
                zo.zoact_multi_forward(ctx, L, X, T, shared, pts, seed, Y)
            torch.cuda.synchronize()
            assert ctx.device_status() == 0
            outs.append(Y)
        assert torch.equal(outs[0], outs[1])             # the K ranges are added in a fixed order
        rnd = {torch.float32: 0.0, torch.bfloat16: 2.0 ** -8, torch.float16: 2.0 ** -11}[ydt]
        err = np.abs(np64(outs[0]) - ref)
        assert np.all(err <= bound + rnd * np.abs(ref)), (ydt, float((err - bound - rnd * np.abs(ref)).max()))


def test_few_rows_two_signs_equal_at_zero_eps(ctx):
    # both signs of a stacked pair with equal inputs go through the same accumulator columns' arithmetic
    d_in, d_out, T, r = 2048, 264, 33, 16
    L, W, U, C = _layer(d_in, d_out, r, "bf16", 300, 1)
    x = normal((T, d_in), 6, DEV, dtype=torch.bfloat16)
    Y = torch.empty(2 * T, d_out, dtype=torch.float32, device=DEV)
    zo.zoact_pair_forward(ctx, L, torch.cat([x, x]), T, False, 0.0, 1, 2, Y)
    torch.cuda.synchronize()
    assert torch.equal(Y[:T], Y[T:])


@pytest.mark.parametrize("wtype,r,T,shared,gated", [("bf16", 1, 5, False, False), ("fp16", 8, 40, True, False),
                                                    ("bf16", 7, 16, False, True), ("int4", 8, 33, False, False),
                                                    ("bf16", 21, 100, False, False)])
def test_lowrank_term_alone(ctx, monkeypatch, wtype, r, T, shared, gated):
    # W = 0 and fp32 outputs (gate: a constant): the low-rank term in six products of three bf16 parts.  Left out are
    # mid lo, lo mid and the parts' own remainders, 4 x 2^-27 of |T||P|; the accumulator truncates each of the steps that
    # hold terms (three a K-block of eight ranks) and aligns its products to about as much: 2^-23 each.  A product that
    # is missing is 2^-9 (hi mid) or 2^-18 (hi lo, mid mid) of |T||P|, far above that.
    monkeypatch.setenv("ZOACT_PAIR_KERNEL", "few")
    d_in, d_out, seed = 128, 264, 3
    dt = torch.float16 if wtype == "fp16" else torch.bfloat16
    X = normal(((T if shared else 2 * T), d_in), 1, DEV, dtype=dt)
    P = normal(((T if shared else 2 * T), r), 2, DEV)
    U = normal((d_in, r), 3, DEV)
    C = normal((d_out * r,), 4, DEV)

    def layer(c, lid):
        if wtype == "int4":
            return zo.make_layer(torch.zeros(d_out, d_in // 2, dtype=torch.uint8, device=DEV), U, c, lid,
                                 w_scales=torch.ones(d_out, 1, dtype=torch.float16, device=DEV), wtype=zo.DT_INT4_G128,
                                 d_in=d_in)
        return zo.make_layer(torch.zeros(d_out, d_in, dtype=dt, device=DEV), U, c, lid)

    Y = torch.empty(2 * T, d_out, device=DEV)
    if gated:
        # the gate's term the constant 20 (one rank of P is 1 there): silu(20) = 20 within 2^-23, the up term under test
        P[:, 0] = 1.0
        Cg = torch.zeros(d_out, r, device=DEV)
        Cg[:, 0] = 20.0
        zo.zoact_pair_forward_gated(ctx, layer(Cg.reshape(-1), 0), layer(C, 1), X, T, shared, 0.0, seed, 1, Y, P_gate=P,
                                    P_up=P)
    else:
        zo.zoact_pair_forward(ctx, layer(C, 0), X, T, shared, 0.0, seed, 1, Y, P=P)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    Pn, Cn = np64(P), np64(C).reshape(d_out, r)
    if shared:
        Pn = np.concatenate([Pn, Pn])
    scale = 20.0 / (1.0 + np.exp(-20.0)) if gated else 1.0
    blocks = (r + 7) // 8
    bound = (4 * 2.0 ** -27 + (6 * blocks) * 2.0 ** -23 + (2.0 ** -21 if gated else 0.0)) * (np.abs(Pn) @ np.abs(Cn).T) * scale
    err = np.abs(np64(Y) - scale * (Pn @ Cn.T))
    assert np.all(err <= bound), float((err / bound).max())
    lost = 2.0 ** -20 * scale * np.abs(Pn) @ np.abs(Cn).T       # what the smallest part is on average
    assert r > 8 or gated or float(err.max()) < float(lost.max())


@pytest.mark.parametrize("wtype,d_in,d_out,T,r,shared,gated", [
    ("bf16", 64, 64, 100, 64, False, False),        # the other route by its estimate
    ("bf16", 256, 512, 64, 16, False, True),
    ("bf16", 256, 512, 100, 64, True, False),       # ... with copies of the shared input
    ("bf16", 256, 512, 128, 64, True, False),       # ... 256 copied rows
    ("int4", 128, 64, 100, 64, False, True),        # ... with W expanded
    ("bf16", 4096, 1024, 16, 16, False, False),     # the few-row kernel
    ("int4", 1024, 264, 245, 16, False, False),     # 490 rows: INT4 in pieces of 240 rows and five, without W expanded
    ("int4", 512, 136, 500, 7, True, False),
    ("int4", 512, 264, 130, 32, False, True),
])
def test_first_call_captured(route, wtype, d_in, d_out, T, r, shared, gated):
    # A first call with the projection given, on a context without scratch, in a capture that may not allocate: the
    # few-row kernel needs no scratch, so it is taken where the other one's is not there.
    L, W, U, C = _layer(d_in, d_out, r, wtype, 100, 3)
    L2 = _layer(d_in, d_out, r, wtype, 200, 4, U=U)[0]
    X = normal(((T if shared else 2 * T), d_in), 5, DEV, dtype=torch.bfloat16)
    P = X.float() @ U
    Y = [torch.zeros(2 * T, d_out, dtype=torch.bfloat16, device=DEV) for _ in range(2)]
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        c = zo.Context(0)
        c.sync_stream()

        def run(y):
            if gated:
                zo.zoact_pair_forward_gated(c, L, L2, X, T, shared, 0.5, 1, 2, y, P_gate=P, P_up=P)
            else:
                zo.zoact_pair_forward(c, L, X, T, shared, 0.5, 1, 2, y, P=P)

        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            run(Y[0])
        g.replay()
        run(Y[1])
        torch.cuda.synchronize()
        assert c.device_status() == 0
    a, b = np64(Y[0]), np64(Y[1])
    assert np.linalg.norm(a - b) <= 2.0 ** -8 * np.linalg.norm(b) and np.abs(a).max() > 0
    c.close()


@pytest.mark.parametrize("T,shared,r,gated,nb", [(245, False, 16, False, 2), (300, True, 16, True, 2), (300, True, 8, False, 3),
                                                 (130, False, 40, True, 2)])
def test_captured_after_a_first_call(T, shared, r, gated, nb):
    # INT4 from 256 rows on W expanded: with the scratch of a first call there a capture takes the same route, same bits
    L, W, U, C = _layer(1024, 264, r, "int4", 100, 3)
    L2 = _layer(1024, 264, r, "int4", 200, 4, U=U)[0]
    pts = [(0.5, 7), (-0.5, 7)] if nb == 2 else [(0.0, 0), (0.25, 1), (0.25, 2)]
    X = normal(((T if shared else nb * T), 1024), 5, DEV, dtype=torch.bfloat16)
    P = X.float() @ U
    Y = [torch.zeros(nb * T, 264, dtype=torch.bfloat16, device=DEV) for _ in range(2)]
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        c = zo.Context(0)
        c.sync_stream()

        def run(y):
            if gated:
                zo.zoact_multi_forward_gated(c, L, L2, X, T, shared, pts, 1, y, P_gate=P, P_up=P)
            else:
                zo.zoact_multi_forward(c, L, X, T, shared, pts, 1, y, P=P)

        run(Y[0])
        torch.cuda.synchronize()
        n = c.launch_count()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            run(Y[1])
        assert c.launch_count() - n == n
        g.replay()
        torch.cuda.synchronize()
    assert torch.equal(Y[0], Y[1])
    c.close()
