"""Measured cases of the CoLA layer library: what a program that trains or
serves LLaMA-style CoLA blocks has it do, through the public entry points of
paper_2502_10940_gb300.cola.

A case is a list of layer groups on one batch of tokens:
  layer      one CoLA layer (o, down, or a lone projection): cola_fwd [+ cola_bwd]
  shared     2 or 3 projections that read one input (gate/up, q/k/v):
             cola_fwd_shared_x [+ cola_bwd_shared_x]
  mlp        the gated MLP: cola_fwd_gate_up, then cola_fwd of the down layer
             [+ cola_bwd_down_gated, then cola_bwd_shared_x of gate/up]
  block      q/k/v, o and the gated MLP of one decoder block, in that order
  recompute  cola_recompute_up: the outputs of `count` projections rebuilt from
             their saved Z (block-level CoLA-M)
The attention, norms and residuals between the groups belong to the caller's
program, so every group reads activations and upstream gradients of its own,
N(0, 1) as after a norm; factors are fan-in Gaussians.  Training groups return
their outputs, everything saved for the backward and every gradient; inference
groups their outputs.

`mode` is "cola", "cola_m" (both: forward + backward) or "infer" (forward
only).  `micro` > 1 accumulates fp32 weight gradients over that many
micro-batches of n tokens, from zero.  `graph`: the pass is captured once and
replayed, as a serving loop does with its decode step.
"""
import math

import torch

from paper_2502_10940_gb300 import cola

BF16 = torch.bfloat16


def _case(kind, n, d, d_ff, r, mode, *, count=1, sigma="silu", micro=1, graph=False, **name):
    return dict(name, kind=kind, n=n, d=d, d_ff=d_ff, r=r, mode=mode, count=count, sigma=sigma, micro=micro, graph=graph)


def listed():
    return [
        # serving, one token for each of 32 sequences through a 1B-shaped block:
        # weight streaming and launch latency; d_ff = 5461 is odd
        _case("block", 32, 2048, 5461, 512, "infer", graph=True, name="decode_1b_block_n32"),
        # serving, one user, one token through a 7B-shaped block
        _case("block", 1, 4096, 11008, 1024, "infer", graph=True, name="decode_7b_block_n1"),
        # a prompt of a few hundred tokens through the q/k/v of a 350M-shaped block
        _case("shared", 509, 1024, 1024, 256, "infer", count=3, name="prompt_350m_qkv_n509"),
        # small-batch training of one 60M-shaped q projection, called eagerly
        _case("layer", 2048, 512, 512, 128, "cola", name="train_60m_q_n2048"),
        # a GELU layer of an odd token count and generic widths, called eagerly
        _case("layer", 3001, 1000, 3000, 192, "cola", sigma="gelu", name="train_gelu_ragged_n3001"),
        # pre-training step of a 60M-shaped block, 256 x 256 tokens: memory-bound
        _case("block", 65536, 512, 1376, 128, "cola", name="train_60m_block"),
        # pre-training step of a 350M-shaped q/k/v group, 512 x 256 tokens
        _case("shared", 131072, 1024, 1024, 256, "cola", count=3, name="train_350m_qkv"),
        # pre-training step of a 1B-shaped gated MLP, 256 x 256 tokens, odd d_ff
        _case("mlp", 65536, 2048, 5461, 512, "cola", name="train_1b_mlp"),
        # two micro-batches of a 1B-shaped o projection into fp32 gradients
        _case("layer", 16384, 2048, 2048, 512, "cola_m", micro=2, name="train_1b_o_accum"),
        # pre-training step of a 7B-shaped gated MLP in CoLA-M, 128 x 256 tokens
        _case("mlp", 32768, 4096, 11008, 1024, "cola_m", name="train_7b_mlp"),
        # batched prompts (32 x 256 tokens) through a 1B-shaped block
        _case("block", 8192, 2048, 5461, 512, "infer", name="prefill_1b_block"),
        # block-level CoLA-M: q/k/v outputs of a 7B-shaped block rebuilt
        _case("recompute", 8192, 4096, 4096, 1024, "cola_m", count=3, name="recompute_7b_qkv"),
    ]


MAX_FLOPS = 9.2e12   # of one drawn pass: no more than the largest listed case
MAX_BYTES = 8.0e9


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    w = _log_int(rng, lo, hi)
    pick = rng.random()
    if pick < 0.4:
        return max(lo, w // 64 * 64)
    if pick < 0.75:
        return max(lo, w // 8 * 8)
    return w


def draw(rng):
    kind = rng.choice(["layer", "layer", "shared", "mlp", "block", "recompute"])
    decode = kind != "recompute" and rng.random() < 0.25
    mode = "infer" if decode else "cola_m" if kind == "recompute" else rng.choice(["cola", "cola", "cola_m", "cola_m", "infer"])
    d = _width(rng, 256, 4096)
    d_ff = _width(rng, 2 * d, 3 * d) if kind != "layer" else _width(rng, max(256, d // 3), 3 * d)
    r = min(16, max(1, round(d / rng.uniform(3.0, 6.0) / 64))) * 64
    n = _log_int(rng, 1, 64) if decode else _log_int(rng, 128, 131072)
    case = _case(kind, n, d, d_ff, r, mode, count=rng.choice([2, 3]) if kind in ("shared", "recompute") else 1,
                 sigma=rng.choice(["silu", "silu", "silu", "gelu", "identity"]),
                 micro=2 if mode in ("cola", "cola_m") and kind in ("layer", "shared") and rng.random() < 0.25 else 1,
                 graph=decode and rng.random() < 0.75)
    while True:
        w = work(case)
        if w["flops"] <= MAX_FLOPS and w["bytes"] <= MAX_BYTES:
            return case
        case["n"] = max(1, int(case["n"] * 0.7))


def _groups(case):
    """(kind, d_in, d_out, projections) of each group, in the order of a pass."""
    k, d, ff = case["kind"], case["d"], case["d_ff"]
    if k == "block":
        return [("proj", d, d, 3), ("proj", d, d, 1), ("mlp", d, ff, 2)]
    return [{"layer": ("proj", d, ff, 1), "shared": ("proj", d, ff, case["count"]), "mlp": ("mlp", d, ff, 2),
             "recompute": ("recompute", d, ff, case["count"])}[k]]


def work(case):
    n, r, train = case["n"], case["r"], case["mode"] != "infer"
    saved = {"cola": 2, "cola_m": 1, "infer": 0}[case["mode"]]
    once = each = flops = 0   # elements per pass, elements per token
    acc = 3 if case["micro"] > 1 else 1   # weight gradients in fp32, zeroed and accumulated: 2 + 2 words against 1
    for kind, a, b, c in _groups(case):
        layers = [(a, b, c)] + ([(b, a, 1)] if kind == "mlp" else [])
        if kind == "recompute":
            each += c * r + c * b
            once += c * r * b
            flops += 2 * r * b * c
            continue
        for di, do, cnt in layers:
            once += cnt * r * (di + do) * (1 + (acc if train else 0))
            each += di + cnt * do + saved * cnt * r
            if train:
                each += cnt * do + di
            flops += (6 if train else 2) * r * (di + do) * cnt
        if kind == "mlp":
            # M = Y_gate * Y_up is written by one call and read by the next;
            # inference stores it alone, training Y_gate, Y_up and M
            each += b if train else -b
    return {"bytes": 2.0 * (once + each * n * case["micro"]), "flops": float(flops) * n * case["micro"]}


# ------------------------------------------------------------------ inputs
def _pitch(w):
    return (w + 7) // 8 * 8


def _empty(rows, cols, dtype=BF16):
    return torch.empty((rows, _pitch(cols)), dtype=dtype, device="cuda")[:, :cols]


class _Random:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def normal(self, rows, cols, std=1.0):
        t = _empty(rows, cols)
        step = max(1, (1 << 28) // max(1, cols))
        for i in range(0, rows, step):
            j = min(rows, i + step)
            v = torch.randn((j - i, cols), generator=self.g, device="cuda")
            t[i:j].copy_(v.mul_(std))
        return t


def _inputs(case, seed):
    """Per group: the factors, and per micro-batch the activations and
    upstream gradients."""
    R = _Random(seed)
    n, r, train = case["n"], case["r"], case["mode"] != "infer"
    out = []
    for kind, a, b, c in _groups(case):
        g = {"kind": kind, "d_in": a, "d_out": b, "count": c}
        g["B"] = [R.normal(b, r, r ** -0.5) for _ in range(c)]
        if kind == "recompute":
            g["Z"] = R.normal(n, c * r)
            out.append(g)
            continue
        g["A"] = R.normal(c * r, a, a ** -0.5)
        g["X"] = [R.normal(n, a) for _ in range(case["micro"])]
        if kind == "mlp":
            g["A2"] = R.normal(r, b, b ** -0.5)
            g["B2"] = R.normal(a, r, r ** -0.5)
            if train:
                g["dY2"] = R.normal(n, a)
        elif train:
            g["dY"] = [[R.normal(n, b) for _ in range(c)] for _ in range(case["micro"])]
        out.append(g)
    return out


# ------------------------------------------------------------- the program
def _prepare_group(case, g):
    n, r, mode = case["n"], case["r"], case["mode"]
    a, b, c, train = g["d_in"], g["d_out"], g["count"], mode != "infer"
    fp32 = case["micro"] > 1
    grad = torch.float32 if fp32 else BF16
    g["d"] = cola.desc(n, a, b, r, ld_x=_pitch(a), ld_y=_pitch(b), ld_a=_pitch(a), sigma=case["sigma"], mode=mode,
                       wgrad_fp32=fp32)
    g["ws"] = cola.workspace(g["d"], c)
    g["Y"] = [_empty(n, b) for _ in range(c)] if train or g["kind"] != "mlp" else [None, None]
    if g["kind"] == "recompute":
        return
    g["Z"] = _empty(n, c * r) if train else None
    g["H"] = _empty(n, c * r) if mode == "cola" else None
    if train:
        g["dX"], g["dA"] = _empty(n, a), _empty(c * r, a, grad)
        g["dB"] = [_empty(b, r, grad) for _ in range(c)]
    if g["kind"] == "mlp":
        g["d2"] = cola.desc(n, b, a, r, ld_x=_pitch(b), ld_y=_pitch(a), ld_a=_pitch(b), sigma=case["sigma"], mode=mode)
        g["ws2"] = cola.workspace(g["d2"])
        g["M"], g["Y2"] = _empty(n, b), _empty(n, a)
        g["Z2"] = _empty(n, r) if train else None
        g["H2"] = _empty(n, r) if mode == "cola" else None
        if train:
            g["dY"] = [_empty(n, b), _empty(n, b)]
            g["dA2"], g["dB2"] = _empty(r, b), _empty(a, r)


def _forward(g, m):
    if g["kind"] == "recompute":
        cola.cola_recompute_up(g["d"], g["Z"], g["B"], g["Y"], g["ws"])
    elif g["kind"] == "mlp":
        cola.cola_fwd_gate_up(g["d"], g["X"][m], g["A"], g["B"][0], g["B"][1], g["M"], g["Y"][0], g["Y"][1], g["Z"],
                              g["H"], g["ws"])
        cola.cola_fwd(g["d2"], g["M"], g["A2"], g["B2"], g["Y2"], g["Z2"], g["H2"], g["ws2"])
    elif g["count"] == 1:
        cola.cola_fwd(g["d"], g["X"][m], g["A"], g["B"][0], g["Y"][0], g["Z"], g["H"], g["ws"])
    else:
        cola.cola_fwd_shared_x(g["d"], g["X"][m], g["A"], g["B"], g["Y"], g["Z"], g["H"], g["ws"])


def _backward(g, m):
    if g["kind"] == "mlp":
        cola.cola_bwd_down_gated(g["d2"], g["M"], g["A2"], g["B2"], g["dY2"], g["Z2"], g["H2"], g["Y"][0], g["Y"][1],
                                 g["dY"][0], g["dY"][1], g["dA2"], g["dB2"], g["ws2"])
        cola.cola_bwd_shared_x(g["d"], g["X"][m], g["A"], g["B"], g["dY"], g["Z"], g["H"], g["dX"], g["dA"], g["dB"],
                               g["ws"])
    elif g["count"] == 1:
        cola.cola_bwd(g["d"], g["X"][m], g["A"], g["B"][0], g["dY"][m][0], g["Z"], g["H"], g["dX"], g["dA"],
                      g["dB"][0], g["ws"])
    else:
        cola.cola_bwd_shared_x(g["d"], g["X"][m], g["A"], g["B"], g["dY"][m], g["Z"], g["H"], g["dX"], g["dA"],
                               g["dB"], g["ws"])


def _pass(state):
    case, groups = state["case"], state["groups"]
    if case["micro"] > 1:
        for g in groups:
            for t in [g["dA"]] + g["dB"]:
                t.zero_()
    for m in range(case["micro"]):
        for g in groups:
            _forward(g, m)
        if case["mode"] != "infer" and case["kind"] != "recompute":
            for g in reversed(groups):
                _backward(g, m)


def _outputs(state):
    outs = []
    for g in state["groups"]:
        o = {"Y": g["Y"]}
        if g["kind"] == "mlp":
            o.update(M=g["M"], Y2=g["Y2"])
        if state["case"]["mode"] != "infer" and g["kind"] != "recompute":
            o.update({k: g[k] for k in ("Z", "H", "dX", "dA", "dB")})
            if g["kind"] == "mlp":
                o.update({k: g[k] for k in ("Z2", "H2", "dY", "dA2", "dB2")})
        outs.append(o)
    return outs


def prepare(case, seed):
    state = {"case": case, "groups": _inputs(case, seed)}
    for g in state["groups"]:
        _prepare_group(case, g)
    if case["graph"]:
        _pass(state)
        torch.cuda.synchronize()
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            _pass(state)
    state["out"] = _outputs(state)
    return state


def run(state):
    if "graph" in state:
        state["graph"].replay()
    else:
        _pass(state)
    return state["out"]


# --------------------------------------------------------------- tolerance
def tolerance(case):
    # bf16 results of up to three chained, bf16-rounded products: measured
    # 1.7e-3 (Z) to 5.7e-3 (the gated MLP's gradients) off the 64-bit values;
    # another summation order moves Z, H, dZ and the results by a last bit
    # here and there.  Single elements of sums that cancel are off by their
    # terms' rounding, some five times that of the whole, against the
    # result's root mean square.
    return {"rel": 1e-2, "max": 0.1}


# ------------------------------------------------------------------- exact
def _sigma(name, z):
    if name == "silu":
        s = torch.sigmoid(z)
        return z * s, s * (1 + z * (1 - s))
    if name == "gelu":
        cdf = 0.5 * torch.erfc(-z * math.sqrt(0.5))
        return z * cdf, cdf + z * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)
    return z, torch.ones_like(z)


def _fwd64(sigma, X, A):
    Z = X @ A.T
    return Z, _sigma(sigma, Z)[0]


def exact(case, seed):
    if work(case)["flops"] > 1.0e13:
        return None
    f, sig, train = torch.Tensor.double, case["sigma"], case["mode"] != "infer"
    outs = []
    for g in _inputs(case, seed):
        r = case["r"]
        cols = [slice(j * r, (j + 1) * r) for j in range(g["count"])]
        B = [f(b) for b in g["B"]]
        if g["kind"] == "recompute":
            outs.append({"Y": [_sigma(sig, f(g["Z"][:, s]))[0] @ b.T for s, b in zip(cols, B)]})
            continue
        A = f(g["A"])
        dA = dB = None
        for m in range(case["micro"]):
            X = f(g["X"][m])
            Z, H = _fwd64(sig, X, A)
            Y = [H[:, s] @ b.T for s, b in zip(cols, B)]
            o = {"Y": Y}
            if g["kind"] == "mlp":
                A2, B2 = f(g["A2"]), f(g["B2"])
                M = Y[0] * Y[1]
                Z2, H2 = _fwd64(sig, M, A2)
                o.update(M=M, Y2=H2 @ B2.T)
                if not train:
                    o["Y"] = [None, None]
            if not train:
                continue
            o.update(Z=Z, H=H if case["mode"] == "cola" else None)
            if g["kind"] == "mlp":
                dY2 = f(g["dY2"])
                dZ2 = (dY2 @ B2) * _sigma(sig, Z2)[1]
                dM = dZ2 @ A2
                dY = [dM * Y[1], dM * Y[0]]
                o.update(Z2=Z2, H2=H2 if case["mode"] == "cola" else None, dY=dY, dA2=dZ2.T @ M, dB2=dY2.T @ H2)
            else:
                dY = [f(t) for t in g["dY"][m]]
            dZ = torch.cat([t @ b for t, b in zip(dY, B)], 1) * _sigma(sig, Z)[1]
            pA, pB = dZ.T @ X, [t.T @ H[:, s] for t, s in zip(dY, cols)]
            dA = pA if dA is None else dA + pA
            dB = pB if dB is None else [x + y for x, y in zip(dB, pB)]
            o.update(dX=dZ @ A, dA=dA, dB=dB)
        outs.append(o)
    return outs
