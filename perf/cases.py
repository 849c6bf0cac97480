"""What the speed of this framework is measured on: the work its users have it do, through its public entry points.

Five kinds of case:

* ``pair``    one adapted linear of a ZO step: the projection P = X U on the prepared basis, then the pair forward
              (both signs; stacked rows, or one input shared by both signs).
* ``gated``   the SiLU-gated gate / up pair of an MLP: one projection (gate and up share a basis), then the gated
              pair forward.
* ``step``    a whole ZO step through ``ZOStep``: pair forwards with their glue, the loss pair, Adam; two-sided, or
              one-sided with q queries.  Graphs: the fp32 toy, the Llama MLP block, decoders of the Llama and OPT stacks.
* ``update``  the end of a ZO step on its own: the loss over the stacked outputs and Adam over every layer's
              coefficients.
* ``basis``   Algorithm 1 for one layer input: the top-r right singular vectors of its calibration activations.

Shapes are those of the workloads in ``synth/configs.py`` (Llama-3-8B, its INT4 form, OPT-13B, the 256-wide toy), the
ranks those of the paper's ablation (1 to 256; 16 and 32 in the workloads), and generic ones.

In ``step`` cases C = 0.3 Z + N(0, 0.01^2) along the step's own perturbation Z and eps = 0.05 (1e-3 in fp32): with the
default eps = 1e-3 and C independent of Z the estimator of a 16-bit step is the rounding noise of its outputs, and no
two implementations would agree on it or on the update it makes.
"""
import math

import torch

import paper_2607_01125_gb300 as zo
from paper_2607_01125_gb300.model import AdaptedLinear, ZOStep, coefficient_offsets

DEV = "cuda:0"
TORCH = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16, "int4": torch.bfloat16}
ACTS = {"none": zo.ACT_NONE, "relu": zo.ACT_RELU, "gelu": zo.ACT_GELU}
SEED, QUERY = 7, 3                     # the step's Philox seed and query id
LR, BETA1, BETA2, ADAM_EPS = 1e-4, 0.9, 0.999, 1e-8

LLAMA = [("q", 4096, 4096), ("k", 4096, 1024), ("v", 4096, 1024), ("o", 4096, 4096), ("gate", 4096, 14336),
         ("up", 4096, 14336), ("down", 14336, 4096)]
OPT = [("q", 5120, 5120), ("k", 5120, 5120), ("v", 5120, 5120), ("o", 5120, 5120), ("fc1", 5120, 20480),
       ("fc2", 20480, 5120)]
RANKS = [1, 4, 8, 16, 16, 16, 32, 32, 64, 128, 256]


def listed():
    return [
        # the smallest program: the two-layer fp32 graph of the workloads, where launches and latency count
        dict(name="toy_step", kind="step", graph="toy", wtype="fp32", T=64, r=8, d=256, queries=0),
        # one short sequence through an attention projection: the frozen weight is read for 32 stacked rows
        dict(name="pair_q_t16", kind="pair", wtype="bf16", d_in=4096, d_out=4096, T=16, r=16, act="none", shared=False),
        # a short prompt through the INT4 down projection at the paper's INT4 rank
        dict(name="pair_int4_down_t64", kind="pair", wtype="int4", d_in=14336, d_out=4096, T=64, r=32, act="none",
             shared=False),
        # one ragged sequence through the gated MLP input
        dict(name="gated_t100", kind="gated", wtype="bf16", d_in=4096, d_out=14336, T=100, r=16, shared=False),
        # an odd batch through OPT's first MLP layer (ReLU fused), rows of one tile in both signs
        dict(name="pair_fc1_fp16_t333", kind="pair", wtype="fp16", d_in=5120, d_out=20480, T=333, r=32, act="relu",
             shared=False),
        # the MLP block's training step as the workload states it (gate and up on a shared input)
        dict(name="mlp_step_t2048", kind="step", graph="mlp", wtype="bf16", T=2048, r=16, queries=0),
        # the paper's own one-sided estimator with 8 queries on the same block
        dict(name="mlp_step_q8_t512", kind="step", graph="mlp", wtype="bf16", T=512, r=16, queries=8),
        # the training step of the full-width stack (two of its 32 decoders) on 16 x 256 tokens
        dict(name="llama_step_t4096", kind="step", graph="llama", wtype="bf16", T=4096, r=16, decoders=2, queries=0),
        # loss and Adam of the full Llama stack: 224 layers, 22.0 M coefficients, 4096 tokens
        dict(name="update_llama", kind="update", graph="llama", layers=32, T=4096, n=4096, r=16, dtype="bf16", queries=0),
        # bases: the widest Llama layer input, OPT's as its workload states it, the ablation's largest rank
        dict(name="basis_down_r16", kind="basis", dtype="bf16", n_tok=512, d=14336, r=16, decay=1.0),
        dict(name="basis_opt_r32", kind="basis", dtype="fp16", n_tok=4096, d=5120, r=32, decay=1.0),
        dict(name="basis_r256", kind="basis", dtype="bf16", n_tok=512, d=4096, r=256, decay=0.5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "gated", "gated", "step", "step", "update", "basis", "basis"])
    if kind == "pair":
        wtype = rng.choice(["bf16", "bf16", "fp16", "int4"])
        if rng.random() < 0.3:         # generic widths
            d_in, d_out = 8 * _log(rng, 32, 1024), 8 * _log(rng, 32, 1024)
            if wtype == "int4":
                d_in = max(128, d_in // 128 * 128)
        else:
            d_in, d_out = rng.choice([s[1:] for s in (OPT if wtype == "fp16" else LLAMA)])
        return dict(kind=kind, wtype=wtype, d_in=d_in, d_out=d_out, T=_log(rng, 16, 4096), r=rng.choice(RANKS),
                    act=rng.choice(["none", "none", "relu"]), shared=rng.random() < 0.25)
    if kind == "gated":
        d_in, d_out = (4096, 14336) if rng.random() < 0.7 else (128 * _log(rng, 2, 48), 8 * _log(rng, 64, 2048))
        return dict(kind=kind, wtype=rng.choice(["bf16", "bf16", "int4"]), d_in=d_in, d_out=d_out,
                    T=_log(rng, 16, 4096), r=rng.choice(RANKS), shared=rng.random() < 0.4)
    if kind == "step":
        graph = rng.choice(["toy", "mlp", "mlp", "llama", "llama", "opt"])
        queries = rng.choice([0, 0, 0, 4, 8])
        if graph == "toy":
            return dict(kind=kind, graph=graph, wtype="fp32", T=_log(rng, 16, 1024), r=rng.choice([1, 4, 8, 16, 32]),
                        d=8 * rng.randint(16, 64), queries=queries)
        wtype = "fp16" if graph == "opt" else "int4" if graph == "llama" and rng.random() < 0.4 else "bf16"
        # one-sided differences of two losses need tokens to stand clear of the outputs' 16-bit rounding
        T = _log(rng, 64, 2048) if queries == 0 else _log(rng, 256, 512)
        c = dict(kind=kind, graph=graph, wtype=wtype, T=T, r=rng.choice([1, 8, 16, 16, 32, 128]), queries=queries)
        if graph != "mlp":
            c["decoders"] = rng.choice([1, 2]) if graph == "llama" else 1
        return c
    if kind == "update":
        graph = rng.choice(["llama", "opt"])
        return dict(kind=kind, graph=graph, layers=_log(rng, 1, 32), T=_log(rng, 16, 4096),
                    n=4096 if graph == "llama" else 5120, r=rng.choice([1, 8, 16, 16]),
                    dtype="fp16" if graph == "opt" else "bf16", queries=rng.choice([0, 0, 8]) if graph == "llama" else 0)
    r = rng.choice([1, 4, 8, 16, 16, 32, 32, 64, 128])
    return dict(kind=kind, dtype=rng.choice(["bf16", "bf16", "fp16"]), n_tok=_log(rng, 400, 4096),
                d=rng.choice([4096, 4096, 5120, 14336, 8 * rng.randint(64, 1000)]), r=r, decay=1.0 if r <= 32 else 0.5)


# ---- inputs ----
_CTX = []


def _ctx():
    """The one library context a program keeps."""
    if not _CTX:
        _CTX.append(zo.Context(0))
    return _CTX[0]


def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1000003 + salt) & 0x7FFFFFFFFFFFFFFF)
    return g


def _randn(g, *shape, std=1.0, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device=DEV).mul_(std).to(dtype)


def _tokens(g, rows, d, dtype, rank=64, noise=0.05, signal=None):
    """Tokens with a rank-`rank` Gaussian signal and a share `noise` of the energy in noise, unit RMS per token."""
    if signal is None:
        signal = _randn(g, rank, d, std=rank ** -0.5)
    x = _randn(g, rows, signal.shape[0]) @ signal * math.sqrt(1 - noise) + _randn(g, rows, d, std=math.sqrt(noise))
    return (x / x.pow(2).mean(dim=1, keepdim=True).sqrt()).to(dtype)


def _basis(g, d, r):
    return torch.linalg.qr(_randn(g, d, r))[0].contiguous()


def _quantize(W):
    """Symmetric INT4 in groups of 128 along d_in: packed nibbles (low nibble first) and fp16 scales."""
    d_out, d_in = W.shape
    Wg = W.reshape(d_out, d_in // 128, 128)
    s = (Wg.abs().amax(dim=2) / 7.0).to(torch.float16)
    q = torch.round(Wg / s.float().clamp_min(1e-12).unsqueeze(2)).clamp_(-8, 7).to(torch.int8).reshape(d_out, d_in)
    nib = (q & 0xF).to(torch.uint8)
    return (nib[:, 0::2] | (nib[:, 1::2] << 4)).contiguous(), s.contiguous()


def _weight(g, d_out, d_in, wtype, std=0.02):
    """(W, scales or None) in the storage of wtype."""
    if wtype == "int4":
        return _quantize(_randn(g, d_out, d_in, std=std))
    return _randn(g, d_out, d_in, std=std, dtype=TORCH[wtype]), None


def _wide(W, scales):
    """The frozen weight in 64 bits."""
    if scales is None:
        return W.double()
    q = torch.stack([W & 0xF, W >> 4], dim=2).reshape(W.shape[0], -1).to(torch.int16)
    q = torch.where(q >= 8, q - 16, q).double()
    return (q.reshape(W.shape[0], -1, 128) * scales.double().unsqueeze(2)).reshape(W.shape[0], -1)


def _specs(case):
    """(name, d_in, d_out) of a graph's adapted linears in forward order."""
    g = case["graph"]
    if g == "toy":
        return [("l1", case["d"], case["d"]), ("l2", case["d"], case["d"])]
    if g == "mlp":
        return [("gate", 4096, 14336), ("up", 4096, 14336), ("down", 14336, 4096)]
    n = case.get("decoders", case.get("layers"))
    return [(f"{L}.{s[0]}", s[1], s[2]) for L in range(n) for s in (LLAMA if g == "llama" else OPT)]


def _input_of(name):
    """The name of the linear whose basis `name` shares (linears that read one input have one basis)."""
    return name.replace(".k", ".q").replace(".v", ".q").replace("up", "gate")


def _d_model(case):
    return {"toy": case.get("d"), "mlp": 4096, "llama": 4096, "opt": 5120}[case["graph"]]


def _shared_rows(case, name):
    return {"toy": name == "l1", "mlp": name != "down"}.get(case["graph"], name in ("0.q", "0.k", "0.v"))


def _prepared(U, wtype):
    """The basis in the projection's operand form, made once as a program does."""
    t = torch.empty(zo.zoact_basis_prepared_bytes(U.shape[0], U.shape[1]), dtype=torch.uint8, device=DEV)
    zo.zoact_basis_prepare(_ctx(), U, zo.TORCH_DT[TORCH[wtype]], t)
    return t


def _layer(W, scales, U, C, layer_id):
    wtype = None if scales is None else zo.DT_INT4_G128
    return zo.make_layer(W, U, C, layer_id, w_scales=scales, wtype=wtype)


def prepare(case, seed):
    return {"pair": _prepare_linear, "gated": _prepare_linear, "step": _prepare_step, "update": _prepare_update,
            "basis": _prepare_basis}[case["kind"]](case, seed)


def _linear_inputs(case, seed):
    g, r, d_in, d_out = _gen(seed), case["r"], case["d_in"], case["d_out"]
    rows = case["T"] if case["shared"] else 2 * case["T"]
    n = 2 if case["kind"] == "gated" else 1
    Ws = [_weight(g, d_out, d_in, case["wtype"]) for _ in range(n)]
    return dict(X=_tokens(g, rows, d_in, TORCH[case["wtype"]]), U=_basis(g, d_in, r), Ws=Ws,
                Cs=[_randn(g, d_out, r, std=0.1) for _ in range(n)])


def _prepare_linear(case, seed):
    s = _linear_inputs(case, seed)
    s["case"], s["ctx"], s["eps"] = case, _ctx(), 0.05
    s["utc"] = _prepared(s["U"], case["wtype"])
    s["layers"] = [_layer(W, sc, s["U"], C, i) for i, ((W, sc), C) in enumerate(zip(s["Ws"], s["Cs"]))]
    s["P"] = torch.empty(s["X"].shape[0], case["r"], device=DEV)
    s["Y"] = torch.empty(2 * case["T"], case["d_out"], dtype=s["X"].dtype, device=DEV)
    return s


def _step_inputs(case, seed):
    g, r, specs = _gen(seed), case["r"], _specs(case)
    dt = TORCH[case["wtype"]]
    std = case["d"] ** -0.5 if case["graph"] == "toy" else 0.02
    offs, bases, lins = coefficient_offsets([_Spec(*s) for s in specs], r), {}, []
    for i, (name, d_in, d_out) in enumerate(specs):
        key = _input_of(name)
        if key not in bases:
            bases[key] = _basis(g, d_in, r)
        W, sc = _weight(g, d_out, d_in, case["wtype"], std)
        lins.append(dict(name=name, W=W, scales=sc, U=bases[key], layer_id=i, offset=offs[i], d_in=d_in, d_out=d_out))
    C = _randn(g, (offs[-1] + specs[-1][2] * r + 3) // 4 * 4, std=0.01)
    for l in lins:
        C[l["offset"]:l["offset"] + l["d_out"] * r] += 0.3 * _normals(SEED, l["layer_id"], QUERY, l["d_out"] * r).float()
    d = _d_model(case)
    x = _tokens(g, case["T"], d, dt, rank=16 if case["graph"] == "toy" else 64)
    target = _randn(g, case["T"], d, dtype=dt) if case["graph"] in ("toy", "mlp") else None
    return lins, C, x, target


class _Spec:
    def __init__(self, name, d_in, d_out):
        self.name, self.d_in, self.d_out = name, d_in, d_out


def _prepare_step(case, seed):
    lins, C, x, target = _step_inputs(case, seed)
    al = [AdaptedLinear(l["name"], l["W"], l["U"], l["layer_id"], l["offset"], case["r"], w_scales=l["scales"],
                        wtype=zo.DT_INT4_G128 if l["scales"] is not None else None, d_in=l["d_in"]) for l in lins]
    kind = {"mlp": "llama_mlp"}.get(case["graph"], case["graph"])
    step = ZOStep(_ctx(), kind, al, case["T"], x.dtype, eps=_step_eps(case), lr=LR,
                  n_queries=case["queries"] or None)
    step.C.copy_(C)
    return dict(case=case, step=step, x=x, target=target, t=0)


def _step_eps(case):
    return 1e-3 if case["graph"] == "toy" else 0.05


def _query(case):
    """ZOStep's query argument of the step whose first query id is QUERY (one-sided: ids query q .. query q + q - 1)."""
    return QUERY if not case["queries"] else 0


def _query_ids(case):
    return [QUERY] if not case["queries"] else list(range(case["queries"]))


def _update_inputs(case, seed):
    g, r = _gen(seed), case["r"]
    specs = _specs(case)
    offs = coefficient_offsets([_Spec(*s) for s in specs], r)
    n = (offs[-1] + specs[-1][2] * r + 3) // 4 * 4
    nb, dt = (case["queries"] + 1 if case["queries"] else 2), TORCH[case["dtype"]]
    y = _randn(g, case["T"], case["n"])
    Y = torch.cat([(y + _randn(g, case["T"], case["n"], std=0.02)).to(dt) for _ in range(nb)])
    blocks = [(o, s[2], r, i) for i, (o, s) in enumerate(zip(offs, specs))]
    C, m = _randn(g, n, std=0.05), _randn(g, n, std=1e-2)
    v = _randn(g, n, std=1e-2).square_()
    return Y, nb, blocks, C, m, v


def _prepare_update(case, seed):
    Y, nb, blocks, C, m, v = _update_inputs(case, seed)
    out = torch.zeros(4 if not case["queries"] else 2 * nb - 1, dtype=torch.float64, device=DEV)
    return dict(case=case, ctx=_ctx(), Y=Y, nb=nb, blocks=blocks, C=C, m=m, v=v, out=out, t=10)


def _calibration(case, seed):
    """Activations whose singular values decay as i^-decay over the signal's rank, plus noise; unit RMS per token."""
    g, rank = _gen(seed), 128 if case["r"] <= 32 else case["r"]
    B = torch.linalg.qr(_randn(g, case["d"], rank))[0].T
    s = torch.arange(1, rank + 1, device=DEV, dtype=torch.float32) ** -case["decay"]
    x = (_randn(g, case["n_tok"], rank) * s * math.sqrt(case["d"])) @ B + _randn(g, case["n_tok"], case["d"], std=0.01)
    return (x / x.pow(2).mean(dim=1, keepdim=True).sqrt()).to(TORCH[case["dtype"]])


def _prepare_basis(case, seed):
    return dict(case=case, ctx=_ctx(), X=_calibration(case, seed), U=torch.empty(case["d"], case["r"], device=DEV),
                evals=torch.empty(min(case["d"], case["r"] + 16), device=DEV))


# ---- one pass ----
def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind in ("pair", "gated"):
        s = state
        zo.zoact_lowrank_proj_prepared(s["ctx"], s["X"], s["utc"], case["r"], s["P"])
        if kind == "pair":
            zo.zoact_pair_forward(s["ctx"], s["layers"][0], s["X"], case["T"], case["shared"], s["eps"], SEED, QUERY,
                                  s["Y"], P=s["P"], act=ACTS[case["act"]])
        else:
            zo.zoact_pair_forward_gated(s["ctx"], s["layers"][0], s["layers"][1], s["X"], case["T"], case["shared"],
                                        s["eps"], SEED, QUERY, s["Y"], P_gate=s["P"], P_up=s["P"])
        return dict(P=s["P"], Y=s["Y"])
    if kind == "step":
        st = state["step"]
        state["t"] += 1
        q = _query(case)
        Y = st.forward(state["x"], SEED, q)
        losses = st.loss(Y, state["target"])
        st.update(state["t"], SEED, q)
        return dict(Y=Y, losses=losses, C=st.C, m=st.m, v=st.v)
    if kind == "update":
        s = state
        s["t"] += 1
        if not case["queries"]:
            zo.zoact_loss_pair(s["ctx"], s["Y"], case["T"], 1e-3, s["out"])
            zo.zoact_adam_step(s["ctx"], s["C"], s["m"], s["v"], s["blocks"], s["out"], LR, BETA1, BETA2, ADAM_EPS,
                               s["t"], SEED, QUERY)
        else:
            zo.zoact_loss_multi(s["ctx"], s["Y"], case["T"], s["nb"], 1e-3, s["out"])
            zo.zoact_adam_step_multi(s["ctx"], s["C"], s["m"], s["v"], s["blocks"], s["out"][s["nb"]:],
                                     _query_ids(case), LR, BETA1, BETA2, ADAM_EPS, s["t"], SEED)
        return dict(losses=s["out"], C=s["C"], m=s["m"], v=s["v"])
    zo.zoact_basis_init(state["ctx"], state["X"], case["r"], state["U"], oversample=16, n_iter=8, seed=5,
                        evals_out=state["evals"])
    return dict(U=state["U"], evals=state["evals"][:case["r"]])


# ---- the work a pass cannot do without ----
def _w_bytes(d_in, d_out, wtype):
    return d_in * d_out * {"fp32": 4.0, "bf16": 2.0, "fp16": 2.0, "int4": 0.5 + 2 / 128}[wtype]


def work(case):
    kind = case["kind"]
    if kind in ("pair", "gated"):
        T, r, d_in, d_out = case["T"], case["r"], case["d_in"], case["d_out"]
        rows, n = (T if case["shared"] else 2 * T), (2 if kind == "gated" else 1)
        b = n * _w_bytes(d_in, d_out, case["wtype"]) + rows * d_in * 2 + 2 * T * d_out * 2 + n * d_out * r * 4 + d_in * r * 4 + rows * r * 4
        return {"bytes": b, "flops": 2.0 * rows * d_in * (n * d_out + r) + n * 2.0 * 2 * T * d_out * r}
    if kind == "step":
        T, r = case["T"], case["r"]
        nb = case["queries"] + 1 if case["queries"] else 2
        es = 4 if case["wtype"] == "fp32" else 2
        b = T * _d_model(case) * es * (1 if case["graph"] not in ("toy", "mlp") else 2) + nb * T * _d_model(case) * es
        f, seen = 0.0, set()
        for name, d_in, d_out in _specs(case):
            rows = T if _shared_rows(case, name) else nb * T
            b += _w_bytes(d_in, d_out, case["wtype"]) + 24.0 * d_out * r
            f += 2.0 * rows * d_in * d_out + 2.0 * nb * T * d_out * r
            if _input_of(name) not in seen:
                seen.add(_input_of(name))
                b += 4.0 * d_in * r
                f += 2.0 * rows * d_in * r
        return {"bytes": b, "flops": f}
    if kind == "update":
        nb, es = (case["queries"] + 1 if case["queries"] else 2), 2
        n = sum(s[2] for s in _specs(case)) * case["r"]
        return {"bytes": float(nb * case["T"] * case["n"] * es + 24 * n), "flops": 6.0 * nb * case["T"] * case["n"] + 20.0 * n}
    # the basis cannot do without reading X and writing U, and without the cheaper of the two products per power step
    n, d, k = case["n_tok"], case["d"], min(case["d"], case["r"] + 16)
    per_step = min(2.0 * d * d * k, 4.0 * n * d * k)
    gram = 2.0 * n * d * d if per_step == 2.0 * d * d * k else 0.0
    return {"bytes": 2.0 * n * d + 4.0 * d * case["r"], "flops": gram + 9 * per_step + 19 * 4.0 * d * k * k}


# ---- tolerances ----
def tolerance(case):
    return TOLERANCE[case["kind"] if case["kind"] != "step" else case["graph"]][case.get("wtype", case.get("dtype"))]


# About four times what a pass differs from exact() by (its error is mostly the rounding of the stored activations) or
# from the same pass with its low-rank term summed in another place.
TOLERANCE = {
    "pair": {"bf16": {"rel": 7e-3, "max": 0.03}, "int4": {"rel": 1.1e-2, "max": 0.05}, "fp16": {"rel": 8e-4, "max": 4e-3}},
    "gated": {"bf16": {"rel": 7e-3, "max": 0.03}, "int4": {"rel": 1.4e-2, "max": 0.2}},
    "toy": {"fp32": {"rel": 3e-5, "max": 1e-3}},
    "mlp": {"bf16": {"rel": 9e-3, "max": 0.06}},
    "llama": {"bf16": {"rel": 3e-2, "max": 0.4}, "int4": {"rel": 3e-2, "max": 0.4}},
    "opt": {"fp16": {"rel": 2e-3, "max": 0.01}},
    "update": {"bf16": {"rel": 1e-6, "max": 1e-5}, "fp16": {"rel": 1e-6, "max": 1e-5}},
    "basis": {"bf16": {"rel": 1.5e-3, "max": 0.06}, "fp16": {"rel": 1.5e-3, "max": 0.06}},
}


# ---- the same results in 64 bits ----
def _normals(seed, layer_id, query, n):
    """The first n normals of a layer's Philox4x32-10 stream, in 64 bits (the uniforms are exact 24-bit values)."""
    M = 0xFFFFFFFF
    g = torch.arange((n + 3) // 4, dtype=torch.int64, device=DEV)
    c = [g & M, torch.full_like(g, layer_id), torch.full_like(g, query & M), torch.full_like(g, query >> 32)]
    k0, k1 = seed & M, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57           # the low 64 bits of the 32 x 32 products
        c = [((p1 >> 32) & M) ^ c[1] ^ k0, p1 & M, ((p0 >> 32) & M) ^ c[3] ^ k1, p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    out = torch.empty(g.numel(), 4, dtype=torch.float64, device=DEV)
    for i in (0, 2):
        u1, u2 = ((c[i] >> 8) + 1).double() * 2.0 ** -24, (c[i + 1] >> 8).double() * 2.0 ** -24
        rad = torch.sqrt(-2.0 * torch.log(u1))
        out[:, i], out[:, i + 1] = rad * torch.cos(2 * math.pi * u2), rad * torch.sin(2 * math.pi * u2)
    return out.reshape(-1)[:n]


def _f32(v):
    return float(torch.tensor(v, dtype=torch.float32))


def _points(case, eps):
    """(coefficient, query id) of every evaluation block."""
    e = _f32(eps)
    if not case.get("queries"):
        return [(e, QUERY), (-e, QUERY)]
    return [(0.0, 0)] + [(e, q) for q in _query_ids(case)]


def _linear64(X, W, U, C, layer_id, T, shared, points):
    """y_b = W x + (C + c_b Z_b)(U^T x) for the stacked blocks b."""
    base, P = X @ W.T, X @ U
    out = []
    for b, (c, q) in enumerate(points):
        rows = slice(0, T) if shared else slice(b * T, (b + 1) * T)
        Cb = C if c == 0.0 else C + c * _normals(SEED, layer_id, q, C.numel()).reshape(C.shape)
        out.append(base[rows] + P[rows] @ Cb.T)
    return torch.cat(out)


def _silu(x):
    return x / (1 + torch.exp(-x))


def _act(x, act):
    return x.clamp_min(0) if act == "relu" else 0.5 * x * (1 + torch.erf(x / math.sqrt(2.0))) if act == "gelu" else x


def _rms(x):
    return x / torch.sqrt(x.pow(2).mean(dim=1, keepdim=True) + 1e-5)


def _adam64(C, m, v, a, blocks, queries, t):
    C, m, v = C.double().clone(), m.double().clone(), v.double().clone()
    b1, b2, lr, ae = _f32(BETA1), _f32(BETA2), _f32(LR), _f32(ADAM_EPS)
    for off, d_out, r, lid in blocks:
        s = slice(off, off + d_out * r)
        g = sum(a[j] * _normals(SEED, lid, q, d_out * r) for j, q in enumerate(queries)) / len(queries)
        m[s] = b1 * m[s] + (1 - b1) * g
        v[s] = b2 * v[s] + (1 - b2) * g * g
        C[s] -= lr / (1 - b1 ** t) * m[s] / (v[s].sqrt() / math.sqrt(1 - b2 ** t) + ae)
    return C, m, v


def _losses64(Y, target, T, nb, eps, one_sided):
    y = [Y[b * T:(b + 1) * T] for b in range(nb)]
    t = 0.0 if target is None else target.double()
    L = [((yb - t) ** 2).mean() for yb in y]
    e = _f32(eps)
    if not one_sided:
        D = ((y[0] - y[1]) * (y[0] + y[1] - 2 * t)).mean()
        return torch.stack(L + [D, D / (2 * e)]), [D / (2 * e)]
    a = [((yb - y[0]) * (yb + y[0] - 2 * t)).mean() / e for yb in y[1:]]
    return torch.stack(L + a), a


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pair", "gated"):
        s = _linear_inputs(case, seed)
        X, U = s["X"].double(), s["U"].double()
        ys = [_linear64(X, _wide(W, sc), U, C.double(), i, case["T"], case["shared"], _points(case, 0.05))
              for i, ((W, sc), C) in enumerate(zip(s["Ws"], s["Cs"]))]
        return dict(P=X @ U, Y=_silu(ys[0]) * ys[1] if kind == "gated" else _act(ys[0], case["act"]))
    if kind == "step":
        return _exact_step(case, seed)
    if kind == "update":
        Y, nb, blocks, C, m, v = _update_inputs(case, seed)
        L, a = _losses64(Y.double(), None, case["T"], nb, 1e-3, bool(case["queries"]))
        C, m, v = _adam64(C, m, v, a, blocks, _query_ids(case), 11)
        return dict(losses=L, C=C, m=m, v=v)
    # eigenvectors of X^T X through the smaller of the two Gram matrices
    X = _calibration(case, seed).double()
    n, d, r = case["n_tok"], case["d"], case["r"]
    if n <= d:
        ev, V = torch.linalg.eigh(X @ X.T)
        ev, V = ev.flip(0)[:r], V.flip(1)[:, :r]
        U = X.T @ V / ev.sqrt()
    elif d <= 6000:
        ev, V = torch.linalg.eigh(X.T @ X)
        ev, U = ev.flip(0)[:r], V.flip(1)[:, :r]
    else:
        return None
    top = U.gather(0, U.abs().argmax(dim=0, keepdim=True))
    return dict(U=U * torch.sign(top), evals=ev)


def _exact_step(case, seed):
    lins, C, x, target = _step_inputs(case, seed)
    by = {l["name"]: l for l in lins}
    T, r, one = case["T"], case["r"], bool(case["queries"])
    pts, rep = _points(case, _step_eps(case)), (4 if case["graph"] == "llama" else 1)

    def lin(name, X, shared):
        l = by[name]
        Cl = C[l["offset"]:l["offset"] + l["d_out"] * r].double().reshape(l["d_out"], r)
        return _linear64(X, _wide(l["W"], l["scales"]), l["U"].double(), Cl, l["layer_id"], T, shared, pts)

    h = x.double()
    if case["graph"] == "toy":
        Y = lin("l2", _act(lin("l1", h, True), "gelu"), False)
    elif case["graph"] == "mlp":
        Y = lin("down", _silu(lin("gate", h, True)) * lin("up", h, True), False)
    else:
        shared = True
        for L in range(case["decoders"]):
            a = _rms(h)
            q, k, v = (lin(f"{L}.{n}", a, shared) for n in "qkv")
            shared = False
            kv = (k + v).reshape(k.shape[0], -1, 128).repeat_interleave(rep, dim=1).reshape(q.shape)
            b = _rms(lin(f"{L}.o", _rms(q + kv), False))
            if case["graph"] == "llama":
                h = lin(f"{L}.down", _rms(_silu(lin(f"{L}.gate", b, False)) * lin(f"{L}.up", b, False)), False)
            else:
                h = lin(f"{L}.fc2", _rms(_act(lin(f"{L}.fc1", b, False), "relu")), False)
        Y = h
    # Losses (with the estimator in them), m and v: none.  The estimator is a small difference of two losses over
    # 2 eps; how far a pass is from its value in 64 bits is the sum of its outputs' roundings, another draw for every
    # order of sums (``update`` cases hold losses and moments to 64 bits on given outputs).  Two-sided, C moves by
    # lr times the sign of a Z; one-sided, its direction is the queries' estimators again.
    _, a = _losses64(Y, target, T, len(pts), _step_eps(case), one)
    z = torch.zeros_like(C)
    Cn, _, _ = _adam64(C, z, z, a, [(l["offset"], l["d_out"], r, l["layer_id"]) for l in lins], _query_ids(case), 1)
    return dict(Y=Y, losses=None, C=None if one else Cn, m=None, v=None)
