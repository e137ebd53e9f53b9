"""The work a user of the library has it do, as cases that can be timed and compared.

A case is a dict of plain values; `kind` says which public entry points it goes through:

  layer  one `hgf.linear_forward` call: a decode token or a prefill batch, optionally behind the LayerNorm
         front end with a gate per head (`ln`), on base-3 weights (`base3`), y in bf16 or fp32
  group  one `hgf.Group` over all projections of `blocks` transformer blocks, each block with weights of its own
         (Q, K and V read one x, the two up-projections another)
  step   the layer calls of one decode step through `blocks` transformer blocks, one after the other: Q, K, V as
         a group (behind their LayerNorms, gates per head), the output projection, the two up-projections as a
         group, the down-projection; captured once as a CUDA graph, as a decode loop does, and replayed.  Each call
         reads an x of its own: what the model computes between the layers (attention, the activation, the
         residual) has left it there
  attn   one `hgf.diff_attention_forward`: the causal differential attention of a prefill or training pass
  train  a training step of one layer: the latent fp32 weights are ternarised and packed, the forward pass
         runs, and the straight-through backward pass gives all five gradients

Layer shapes, ranks and token counts are those of `paper_2602_05269_b200.inputs.CONFIGS` and of bench.py, and odd
sizes around them.
"""
from __future__ import annotations

import math

import torch

from paper_2602_05269_b200 import hgf
from paper_2602_05269_b200.inputs import LayerShape

DEV = "cuda"


def _block(d, ffn, r):
    """The seven projections of a transformer block (those of inputs.CONFIGS)."""
    return [*(LayerShape(n, d, d, r) for n in ("q", "k", "v", "o")), LayerShape("up", d, ffn, r), LayerShape("gate", d, ffn, r),
            LayerShape("down", ffn, d, r)]


def _layer(name, M, K, N, r, *, bf16=True, ln=False, base3=False):
    return {"name": name, "kind": "layer", "M": M, "K": K, "N": N, "r": r, "bf16": bf16, "ln": ln, "base3": base3}


def listed():
    return [
        # The smallest configuration, four tokens: a call whose time is launches, latency and host work.
        _layer("layer_512_m4", 4, 512, 512, 16, bf16=False),
        # The layers of one decode step through eight 1.2B-class blocks for one sequence: the chain that sets the time per token.
        {"name": "step_2048_m1", "kind": "step", "M": 1, "d": 2048, "ffn": 5632, "r": 32, "blocks": 8, "ln": True},
        # All 252 projections of a 1.2B-class model at one token: the packed-weight stream (bench.py's headline).
        {"name": "group_2048_m1", "kind": "group", "M": 1, "d": 2048, "ffn": 5632, "r": 32, "blocks": 36, "bf16": False, "base3": False},
        # The same block at the largest decode batch: sixteen sequences served together.
        {"name": "group_2048_m16", "kind": "group", "M": 16, "d": 2048, "ffn": 5632, "r": 32, "blocks": 36, "bf16": False, "base3": False},
        # 7B-class blocks with weights kept at 1.6 bits, where memory is what is short.
        {"name": "group_4096_b3_m1", "kind": "group", "M": 1, "d": 4096, "ffn": 11008, "r": 64, "blocks": 8, "bf16": True, "base3": True},
        # Prefill of a short prompt through a down-projection: few output tiles, a long contraction.
        _layer("prefill_5632_2048_m512", 512, 5632, 2048, 32),
        # Prefill of a ragged batch through an attention projection with the reference module's front end.
        _layer("prefill_ln_2048_m2000", 2000, 2048, 2048, 32, ln=True),
        # Prefill of a full batch through an up-projection (bench.py's prefill half).
        _layer("prefill_2048_5632_m8192", 8192, 2048, 5632, 32),
        # The same for a 7B-class layer with the widest correction.
        _layer("prefill_4096_11008_m4096", 4096, 4096, 11008, 64),
        # Differential attention over full-length sequences (bench.py's case).
        {"name": "attn_64_l4096", "kind": "attn", "B": 4, "L": 4096, "h": 16, "dh": 64, "bf16": True},
        # Wide heads, ragged length, output kept in fp32.
        {"name": "attn_128_l1500", "kind": "attn", "B": 2, "L": 1500, "h": 16, "dh": 128, "bf16": False},
        # One layer's training step on a full batch (bench.py's backward case, with its forward and its packing).
        {"name": "train_2048_5632_m8192", "kind": "train", "M": 8192, "K": 2048, "N": 5632, "r": 32},
    ]


# ---- drawn cases ------------------------------------------------------------------------------------------
_MAX_LAYER = 4096 * 4096 * 11008       # multiply-adds of the largest listed prefill
_MAX_GROUP = 36 * (4 * 2048 * 2048 + 3 * 2048 * 5632)  # weights of the largest listed group
_MAX_STEP = 8 * (4 * 2048 * 2048 + 3 * 2048 * 5632)
_MAX_ATTN = 4 * 16 * 4096 * 4096 * 64
_MAX_TRAIN = 8192 * 2048 * 5632


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "layer", "group", "group", "step", "attn", "attn", "train"])
    while True:
        if kind == "layer":
            c = {"kind": kind, "M": _log_int(rng, 1, 8192), "K": _log_int(rng, 512, 11008, 64), "N": _log_int(rng, 512, 11008, 8),
                 "r": rng.choice([0, 16, 32, 32, 48, 64]), "bf16": rng.random() < 0.7, "ln": rng.random() < 0.25, "base3": False}
            c["base3"] = rng.random() < 0.15
            if c["M"] * c["K"] * c["N"] <= _MAX_LAYER:
                return c
        elif kind == "group":
            c = {"kind": kind, "M": rng.choice([1, 1, 2, 3, 4, 6, 8, 8, 11, 16]), "d": _log_int(rng, 512, 4096, 64),
                 "ffn": _log_int(rng, 1024, 11008, 64), "r": rng.choice([16, 32, 48, 64]), "blocks": _log_int(rng, 1, 36),
                 "bf16": rng.random() < 0.5, "base3": rng.random() < 0.2}
            # (a group holds problems whose activations fit shared memory, as hgf.h says)
            if c["blocks"] * (4 * c["d"] ** 2 + 3 * c["d"] * c["ffn"]) <= _MAX_GROUP and (c["M"] + 1) * (c["ffn"] + 384) <= 100000:
                return c
        elif kind == "step":
            c = {"kind": kind, "M": _log_int(rng, 1, 16), "d": _log_int(rng, 512, 4096, 64), "ffn": _log_int(rng, 1024, 11008, 64),
                 "r": rng.choice([16, 32, 48, 64]), "blocks": rng.randint(1, 8), "ln": rng.random() < 0.5}
            if c["blocks"] * (4 * c["d"] ** 2 + 3 * c["d"] * c["ffn"]) <= _MAX_STEP:
                return c
        elif kind == "attn":
            c = {"kind": kind, "B": rng.randint(1, 8), "L": _log_int(rng, 64, 8192), "h": rng.choice([4, 8, 12, 16, 32]),
                 "dh": rng.choice([64, 64, 128]), "bf16": rng.random() < 0.7}
            if c["B"] * c["h"] * c["L"] ** 2 * c["dh"] <= _MAX_ATTN:
                return c
        else:
            c = {"kind": kind, "M": _log_int(rng, 64, 8192), "K": _log_int(rng, 512, 8192, 64), "N": _log_int(rng, 512, 8192, 8),
                 "r": rng.choice([0, 16, 32, 64])}
            if c["M"] * c["K"] * c["N"] <= _MAX_TRAIN:
                return c


# ---- inputs -----------------------------------------------------------------------------------------------
# The distributions of paper_2602_05269_b200.inputs, drawn on the device: weights N(0, 0.02), activations N(0, 1) with
# two per cent of outlier channels twenty times as large, A and B scaled by their contraction, gates in (0, 1).
class _Rand:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed) * 1000003 + 17)

    def normal(self, shape, std=1.0, dtype=torch.float32):
        return (torch.randn(shape, generator=self.g, device=DEV) * std).to(dtype)

    def x(self, M, K):
        x = torch.randn((M, K), generator=self.g, device=DEV)
        ch = torch.randperm(K, generator=self.g, device=DEV)[: int(0.02 * K)]
        x[:, ch] *= 20.0
        return x.to(torch.bfloat16)

    def gate(self, n):
        return torch.rand(n, generator=self.g, device=DEV)

    def latent(self, K, N, r, gates=None):
        """A layer's fp32 weights and its correction."""
        w = {"W": self.normal((N, K), 0.02), "At": None, "Bt": None, "gate": None}
        if r:
            w["At"] = self.normal((r, K), K ** -0.5, torch.float16)
            w["Bt"] = self.normal((N, r), r ** -0.5, torch.float16)
            w["gate"] = self.gate(gates or N)
        return w

    def weights(self, K, N, r, base3=False, gates=None):
        """A layer's packed weights and correction, as keyword values of the calls."""
        w = self.latent(K, N, r, gates)
        packed, gamma = hgf.pack_ternary(w.pop("W"), base3=base3)
        return {"packed": packed, "gamma": gamma, **w}

    def norm(self, K):
        return {"ln_weight": 1.0 + self.normal((K,), 0.1), "ln_bias": self.normal((K,), 0.1)}


def _head(N):
    """Channels per gate of the grouped gate: heads of 64 where they divide the width, else one gate for all."""
    return 64 if N % 64 == 0 else N


def _flags(c):
    return (hgf.FLAG_OUT_BF16 if c["bf16"] else 0) | (hgf.FLAG_BASE3 if c["base3"] else 0)


def _prepare_layer(c, rand):
    M, K, N, r, flags = c["M"], c["K"], c["N"], c["r"], _flags(c)
    heads = _head(N) if c["ln"] else None
    s = {"x": rand.x(M, K), "w": rand.weights(K, N, r, c["base3"], -(-N // heads) if heads else None), "flags": flags, "fe": {}}
    if c["ln"]:
        s["fe"] = {**rand.norm(K), "eps": 1e-5, "gate_group": heads}
    s["y"] = torch.empty((M, N), dtype=torch.bfloat16 if c["bf16"] else torch.float32, device=DEV)
    s["ws"] = torch.empty(hgf.workspace_bytes(M, K, N, r, flags), dtype=torch.uint8, device=DEV)
    return s


def _run_layer(c, s):
    w = s["w"]
    return hgf.linear_forward(s["x"], w["packed"], w["gamma"], c["K"], c["N"], w["At"], w["Bt"], w["gate"], y=s["y"],
                              workspace=s["ws"], flags=s["flags"], **s["fe"])


def _prepare_group(c, rand):
    M, shapes = c["M"], _block(c["d"], c["ffn"], c["r"])
    y = torch.empty(c["blocks"] * M * sum(p.d_out for p in shapes), dtype=torch.bfloat16 if c["bf16"] else torch.float32, device=DEV)
    problems, at = [], 0
    for _ in range(c["blocks"]):
        xs = {"q": rand.x(M, c["d"]), "o": rand.x(M, c["d"]), "up": rand.x(M, c["d"]), "down": rand.x(M, c["ffn"])}
        xs["k"] = xs["v"] = xs["q"]
        xs["gate"] = xs["up"]
        for p in shapes:
            n = M * p.d_out
            problems.append({"x": xs[p.name], "d_in": p.d_in, "d_out": p.d_out, "y": y[at:at + n].view(M, p.d_out),
                             **rand.weights(p.d_in, p.d_out, p.r, c["base3"])})
            at += n
    return {"group": hgf.Group(problems, flags=_flags(c)), "y": y}


def _run_group(c, s):
    s["group"].forward()
    return s["y"]


def _prepare_step(c, rand):
    M, d, ffn, r, flags = c["M"], c["d"], c["ffn"], c["r"], hgf.FLAG_OUT_BF16
    out = lambda n: torch.empty((M, n), dtype=torch.bfloat16, device=DEV)  # noqa: E731
    calls, ys, keep = [], [], []

    def single(w, K, N):
        xin, y, ws = rand.x(M, K), out(N), torch.empty(hgf.workspace_bytes(M, K, N, r, flags), dtype=torch.uint8, device=DEV)
        calls.append(lambda: hgf.linear_forward(xin, w["packed"], w["gamma"], K, N, w["At"], w["Bt"], w["gate"], y=y, workspace=ws, flags=flags))
        keep.append((xin, w, ws))
        return y

    def group(N, n, ln):
        xin, problems = rand.x(M, d), []
        for _ in range(n):
            p = {"x": xin, "d_in": d, "d_out": N, "y": out(N), **rand.weights(d, N, r, gates=N // 64 if ln else None)}
            if ln:
                p.update({**rand.norm(d), "eps": 1e-5, "gate_group": 64})
            problems.append(p)
        g = hgf.Group(problems, flags=flags)
        calls.append(g.forward)
        keep.append(g)
        return [p["y"] for p in problems]

    for _ in range(c["blocks"]):
        ys += group(d, 3, c["ln"])
        ys.append(single(rand.weights(d, d, r), d, d))
        ys += group(ffn, 2, False)
        ys.append(single(rand.weights(ffn, d, r), ffn, d))

    def step():
        for call in calls:
            call()

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    return {"graph": graph, "ys": ys, "keep": keep}


def _run_step(c, s):
    s["graph"].replay()
    return s["ys"]


def _prepare_attn(c, rand):
    rows, d = c["B"] * c["L"], c["h"] * c["dh"]
    return {"q": rand.normal((rows, 2 * d), 1.0, torch.bfloat16), "k": rand.normal((rows, 2 * d), 1.0, torch.bfloat16),
            "v": rand.normal((rows, d), 1.0, torch.bfloat16), "lam": hgf.diff_lambda0(c["dh"]),
            "out": torch.empty((rows, d), dtype=torch.bfloat16 if c["bf16"] else torch.float32, device=DEV)}


def _run_attn(c, s):
    return hgf.diff_attention_forward(s["q"], s["k"], s["v"], c["B"], c["L"], c["h"], c["dh"], s["lam"], out=s["out"],
                                      flags=hgf.FLAG_OUT_BF16 if c["bf16"] else 0)


def _prepare_train(c, rand):
    M, K, N, r = c["M"], c["K"], c["N"], c["r"]
    s = {"W": rand.normal((N, K), 0.02), "x": rand.x(M, K), "dy": rand.normal((M, N), 1.0, torch.bfloat16), "At": None, "Bt": None, "gate": None}
    shapes = {"dx": (M, K), "dW": (N, K)}
    if r:
        s["At"], s["Bt"], s["gate"] = rand.normal((r, K), K ** -0.5, torch.float16), rand.normal((N, r), r ** -0.5, torch.float16), rand.gate(N)
        shapes.update({"dAt": (r, K), "dBt": (N, r), "dgate": (N,)})
    s["grads"] = {n: torch.empty(v, device=DEV) for n, v in shapes.items()}
    s["y"] = torch.empty((M, N), dtype=torch.bfloat16, device=DEV)
    s["ws"] = torch.empty(hgf.workspace_bytes(M, K, N, r, hgf.FLAG_OUT_BF16), dtype=torch.uint8, device=DEV)
    s["bws"] = torch.empty(hgf.backward_workspace_bytes(M, K, N, r), dtype=torch.uint8, device=DEV)
    return s


def _run_train(c, s):
    K, N = c["K"], c["N"]
    packed, gamma = hgf.pack_ternary(s["W"])
    y = hgf.linear_forward(s["x"], packed, gamma, K, N, s["At"], s["Bt"], s["gate"], y=s["y"], workspace=s["ws"], flags=hgf.FLAG_OUT_BF16)
    g = hgf.linear_backward(s["x"], packed, gamma, K, N, s["dy"], s["At"], s["Bt"], s["gate"], out=s["grads"], workspace=s["bws"])
    return {"y": y, **{n: g[n] for n in s["grads"]}}


_KINDS = {"layer": (_prepare_layer, _run_layer), "group": (_prepare_group, _run_group), "step": (_prepare_step, _run_step),
          "attn": (_prepare_attn, _run_attn), "train": (_prepare_train, _run_train)}


def prepare(case, seed):
    return {"case": case, **_KINDS[case["kind"]][0](case, _Rand(seed))}


def run(state):
    return _KINDS[state["case"]["kind"]][1](state["case"], state)


# ---- the same in 64 bits ----------------------------------------------------------------------------------
# The quantisers decide in the precision that defines them (binary32 scales); every product and sum is a double's.
def _ternary(W):
    """(gamma_W as the nearest binary32 value, codes): the codes are those whose weight is nearest gamma_W times them."""
    gamma = W.double().abs().mean().float().double()
    return gamma, (W.double() > 0.5 * gamma).double() - (W.double() < -0.5 * gamma).double()


def _dequantised(x, norm=None):
    """The int8 values times their scale, as doubles."""
    if norm is None:
        g = x.double().abs().amax(1, keepdim=True).clamp_min(float(torch.tensor(1e-5)))
        return torch.round(127.0 * x.double() / g).clamp(-127, 127) * g / 127.0
    xd = x.double()
    mean, var = xd.mean(1, keepdim=True), xd.var(1, unbiased=False, keepdim=True)
    n = (x.float() - mean.float()) * (var + 1e-5).rsqrt().float() * norm["ln_weight"] + norm["ln_bias"]
    g = n.abs().amax(1, keepdim=True).clamp_min(1e-5)
    return torch.round(n * (127.0 / g)).clamp(-127, 127).double() * g.double() / 127.0


def _exact_layer(x, w, norm=None, heads=1):
    gamma, T = _ternary(w["W"])
    y = _dequantised(x, norm) @ T.T * gamma
    if w["At"] is not None:
        z = x.double() @ w["At"].double().T
        n = torch.arange(T.shape[0], device=DEV) // heads
        y += (z * torch.sigmoid(z)) @ w["Bt"].double().T * w["gate"].double()[n]
    return y


def _exact_attn(c, rand):
    B, L, h, dh = c["B"], c["L"], c["h"], c["dh"]
    q, k, v = (rand.normal((B * L, n), 1.0, torch.bfloat16) for n in (2 * h * dh, 2 * h * dh, h * dh))
    lam = 0.8 - 0.6 * math.exp(-0.3 * dh)
    q, k, v = q.view(B, L, 2, h, dh), k.view(B, L, 2, h, dh), v.view(B, L, h, dh)
    out = torch.empty((B, L, h, dh), dtype=torch.float64, device=DEV)
    for b in range(B):
        for hd in range(h):
            for i in range(0, L, 2048):  # rows of the score matrix at a time
                e = min(L, i + 2048)
                future = torch.ones((e - i, e), dtype=torch.bool, device=DEV).triu(i + 1)
                p = [torch.softmax((q[b, i:e, s, hd].double() @ k[b, :e, s, hd].double().T * dh ** -0.5).masked_fill(future, -math.inf), 1)
                     for s in (0, 1)]
                out[b, i:e, hd] = (p[0] - lam * p[1]) @ v[b, :e, hd].double()
    return out.view(B * L, h * dh)


def _exact_train(c, rand):
    M, K, N, r = c["M"], c["K"], c["N"], c["r"]
    W, x, dy = rand.normal((N, K), 0.02), rand.x(M, K), rand.normal((M, N), 1.0, torch.bfloat16).double()
    w = {"W": W, "At": None}
    if r:
        w = {"W": W, "At": rand.normal((r, K), K ** -0.5, torch.float16), "Bt": rand.normal((N, r), r ** -0.5, torch.float16), "gate": rand.gate(N)}
    gamma, T = _ternary(W)
    out = {"y": _exact_layer(x, w), "dx": dy @ T * gamma, "dW": dy.T @ _dequantised(x)}
    if r:
        A, B, g, x = w["At"].double(), w["Bt"].double(), w["gate"].double(), x.double()
        z = x @ A.T
        s = torch.sigmoid(z)
        dz = ((dy * g) @ B) * (s * (1 + z * (1 - s)))
        hy = dy.T @ (z * s)
        out["dx"] += dz @ A
        out.update({"dAt": dz.T @ x, "dBt": hy * g[:, None], "dgate": (hy * B).sum(1)})
    return out


def exact(case, seed):
    """What run() gives, from the same inputs (drawn in the order in which prepare() draws them)."""
    c, rand = case, _Rand(seed)
    if c["kind"] == "attn":
        return _exact_attn(c, rand)
    if c["kind"] == "train":
        return _exact_train(c, rand)
    if c["kind"] == "layer":
        M, K, N, r = c["M"], c["K"], c["N"], c["r"]
        heads = _head(N) if c["ln"] else 1
        x, w = rand.x(M, K), rand.latent(K, N, r, -(-N // heads) if c["ln"] else None)
        return _exact_layer(x, w, rand.norm(K) if c["ln"] else None, heads)
    M, d, ffn, r, ys = c["M"], c["d"], c["ffn"], c["r"], []
    if c["kind"] == "group":
        for _ in range(c["blocks"]):
            xs = {"q": rand.x(M, d), "o": rand.x(M, d), "up": rand.x(M, d), "down": rand.x(M, ffn)}
            xs["k"] = xs["v"] = xs["q"]
            xs["gate"] = xs["up"]
            for p in _block(d, ffn, r):
                ys.append(_exact_layer(xs[p.name], rand.latent(p.d_in, p.d_out, p.r)).flatten())
        return torch.cat(ys)
    for _ in range(c["blocks"]):
        for N, n, ln in ((d, 3, c["ln"]), (ffn, 2, False)):
            x = rand.x(M, d)
            for _ in range(n):
                w = rand.latent(d, N, r, N // 64 if ln else None)
                ys.append(_exact_layer(x, w, rand.norm(d) if ln else None, 64 if ln else 1))
            K = d if n == 3 else ffn  # the output projection, the down-projection
            w = rand.latent(K, d, r)
            ys.append(_exact_layer(rand.x(M, K), w))
    return ys


# ---- work and tolerance -----------------------------------------------------------------------------------
def _layer_work(M, p: LayerShape, ybytes, base3=False):
    """Bytes of the weights, the correction, the gate, x and y once each; the products as multiply and add."""
    K, N, r = p.d_in, p.d_out, p.r
    weights = K * N / 5 if base3 else K * N / 4
    return (weights + (2 * r * (K + N) + 4 * N if r else 0) + 2 * M * K + ybytes * M * N, 2 * M * K * N + 2 * M * r * (K + N))


def work(case):
    c = case
    if c["kind"] == "layer":
        b, f = _layer_work(c["M"], LayerShape("", c["K"], c["N"], c["r"]), 2 if c["bf16"] else 4, c["base3"])
    elif c["kind"] in ("group", "step"):
        ybytes = 2 if c["kind"] == "step" or c["bf16"] else 4
        per = [_layer_work(c["M"], p, ybytes, c.get("base3", False)) for p in _block(c["d"], c["ffn"], c["r"])]
        # K, V and the second up-projection read an x that is counted with Q and the first
        b = c["blocks"] * (sum(x for x, _ in per) - 3 * 2 * c["M"] * c["d"])
        f = c["blocks"] * sum(x for _, x in per)
    elif c["kind"] == "attn":
        rows, d = c["B"] * c["L"], c["h"] * c["dh"]
        b = rows * d * (2 * 2 + 2 * 2 + 2 + (2 if c["bf16"] else 4))
        # two streams, two products each, over the visible half of the score matrix
        f = 2 * 2 * 2 * c["B"] * c["h"] * (c["L"] * (c["L"] + 1) / 2) * c["dh"]
    else:
        M, K, N, r = c["M"], c["K"], c["N"], c["r"]
        # read: W, x, dy, A, B, gate; written: y, dx, dW and the small gradients
        b = 4 * N * K + 2 * M * K + 2 * M * N + 2 * M * N + 4 * M * K + 4 * N * K + (6 * r * (K + N) + 8 * N if r else 0)
        f = 3 * 2 * M * K * N + (2 * M * r * (K + N) * 3 if r else 0)
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    """About four times what the library shows against the same path in 64 bits (relative 2-norm): decode outputs in
    fp32 7e-7; outputs rounded to bf16 1.7e-3; fp32 outputs of the tensor-core path, whose correction is rounded to
    fp16, 3e-4 (and the LayerNorm's last bit can move a code by one); attention 2.5e-3 (probabilities and output in
    bf16, two streams that partly cancel); gradients of bf16 products up to 3e-3."""
    c = case
    if c["kind"] == "attn":
        return {"rel": 1e-2}
    if c["kind"] == "train":
        return {"rel": 1.2e-2}
    if c["kind"] == "step" or c["bf16"]:
        return {"rel": 6e-3}
    if c["kind"] == "layer" and (c["M"] > hgf.DECODE_MAX_M or c["ln"]):
        return {"rel": 1.2e-3}
    return {"rel": 1e-5}
