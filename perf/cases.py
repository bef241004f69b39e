"""The measured cases of the NOBLE linear layer, through its public entry points.

A case is one call, or one forward and backward, of a layer as a program uses
it: ``binding.forward`` / ``binding.backward`` on buffers and parameters that
the program keeps, or one fused optimizer step.  Kinds:

    "step"   forward, then backward: y, dx and every parameter gradient
    "infer"  forward with NOBLE_FLAG_INFERENCE: y
    "adamw"  one noble_adamw_step over a layer's parameters: the new
             parameters, their bf16 copies and both moments

Sizes are those of the package's configurations (inputs.py) or generic ones of
the same ranges.
"""
from __future__ import annotations

import math

import torch

from paper_2603_06492_gb300 import binding
from paper_2603_06492_gb300.inputs import geglu_hidden

SIGMAS = ("cosnet", "cos1", "identity", "tanh1", "tanh2", "leaky1", "leaky2", "gelu1", "gelu2", "cos3")
RANKS = (0, 16, 32, 64, 128, 256)


def _case(kind, T, d_in, d_out, r, dtype="bf16", sigma="cosnet", name=None):
    c = {"kind": kind, "T": T, "d_in": d_in, "d_out": d_out, "r": r, "dtype": dtype, "sigma": sigma}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest configuration: checking a change of a model in fp32,
        # where launches and their gaps are all there is
        _case("step", 256, 128, 128, 16, "fp32", name="fp32-tiny-step"),
        # the fp32 mode on one 1024-token sequence of the 1024-wide decoder:
        # a run that a bf16 training run is compared with
        _case("step", 1024, 1024, 1024, 64, "fp32", name="fp32-sequence-step"),
        # generating with a 2048-wide decoder: one token of each of 24 sequences
        _case("infer", 24, 2048, 6144, 128, name="decode-24-qkv"),
        # reading a prompt of one 1024-token sequence, 1024-wide decoder
        _case("infer", 1024, 1024, 4096, 64, name="prefill-1024-ffn-up"),
        # fine-tuning a ViT on small batches: eight images of 197 tokens
        _case("step", 8 * 197, 768, 2304, 32, name="vit-8-images-qkv-step"),
        # training the 1024-wide decoder: its smallest and its widest projection
        _case("step", 8192, 1024, 1024, 64, name="base-attn-out-step"),
        _case("step", 8192, 1024, 4096, 64, name="base-ffn-up-step"),
        # its GeGLU FFN on packed text of no particular length
        _case("step", 7001, 1024, geglu_hidden(1024), 64, name="base-geglu-ragged-step"),
        # training a ViT with 256 images, at the widest bottleneck
        _case("step", 256 * 197, 768, 2304, 256, name="vit-256-images-r256-step"),
        # the ablation's deepest bottleneck, through its own entry points
        _case("step", 4096, 2048, 2048, 128, sigma="cos3", name="ablation-cos3-step"),
        # training the 2048-wide decoder: its largest projection
        _case("step", 16384, 2048, 8192, 128, name="large-ffn-up-step"),
        # the optimizer step of that projection's parameters
        _case("adamw", 0, 2048, 8192, 128, name="adamw-large-ffn-up"),
    ]


def _flops(c):
    """Multiply-adds times two of one pass (contractions only)."""
    T, di, do, r = c["T"], c["d_in"], c["d_out"], c["r"]
    mats = {"cosnet": 1, "tanh2": 1, "leaky2": 1, "gelu2": 1, "cos3": 2}.get(c["sigma"], 0)
    one = 2.0 * T * (di * do + r * (di + do) + mats * r * r)
    return {"step": 3.0, "infer": 1.0, "adamw": 0.0}[c["kind"]] * one


# the largest drawn pass: the largest listed one in bf16; on the fp32 path,
# whose rate is that of the CUDA cores, one of about that duration
_MOST = {"bf16": 1.7e12, "fp32": 8e9}


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _width(rng, lo, hi):
    w = _log_uniform(rng, lo, hi)
    q = rng.choice((8, 64, 64, 128))  # widths are multiples of 8; most models' of 64
    return max(lo, int(w / q + 0.5) * q)


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "infer", "infer", "adamw"))
    if kind == "adamw":
        return _case(kind, 0, _width(rng, 128, 2048), _width(rng, 128, 8192), rng.choice(RANKS))
    dtype = "fp32" if kind == "step" and rng.random() < 0.2 else "bf16"
    sigma = "cosnet" if rng.random() < 0.65 else rng.choice(SIGMAS[1:])
    for _ in range(1000):
        hi = 4096 if dtype == "fp32" else 50432 if kind == "step" else 16384
        # generation handles a few tokens a call, all other uses whole sequences
        lo = 64 if kind == "step" else 1
        c = _case(kind, int(_log_uniform(rng, lo, hi)), _width(rng, 128, 8192), _width(rng, 128, 8192),
                  rng.choice(RANKS), dtype, sigma)
        # a bottleneck is narrower than the layer
        if c["r"] <= min(c["d_in"], c["d_out"]) // 2 and _flops(c) <= _MOST[dtype]:
            if c["r"] == 0:
                c["sigma"] = "cosnet"  # a plain layer has no bottleneck
            return c
    return _case("step", 1000, 512, 512, 32)


# ---------------------------------------------------------------- inputs
def _names(c):
    """Parameters that the case's layer has."""
    out = ["W", "bias"]
    if c["r"]:
        s = c["sigma"]
        out += ["W_down", "W_up"]
        if s in ("cosnet", "cos1", "cos3"):
            out += ["omega1", "phi1"]
        if s in ("cosnet", "cos3"):
            out += ["omega2", "phi2"]
        if s in ("cosnet", "cos3", "tanh2", "leaky2", "gelu2"):
            out += ["M"]
        if s == "cos3":
            out += ["M2", "omega3", "phi3"]
    return out


def _shape(c, name):
    di, do, r = c["d_in"], c["d_out"], c["r"]
    return {"W": (do, di), "bias": (do,), "W_down": (r, di), "W_up": (do, r), "M": (r, r), "M2": (r, r)}.get(name, (r,))


def _tensors(c, seed):
    """x, dy and the parameters, in the distributions of inputs.py."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    tdt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32

    def normal(shape, std, dtype):
        return (torch.randn(shape, generator=g, device="cuda") * std).to(dtype)

    def uniform(shape, lo, hi):
        return torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo

    p = {}
    for n in _names(c):
        s = _shape(c, n)
        if n in ("W", "W_down"):
            p[n] = normal(s, 1.0 / math.sqrt(c["d_in"]), tdt)
        elif n == "W_up":
            p[n] = normal(s, 0.02, tdt)
        elif n == "bias":
            p[n] = normal(s, 0.02, torch.float32)
        elif n in ("M", "M2"):
            p[n] = normal(s, 1.0 / math.sqrt(c["r"]), torch.float32)
        elif n.startswith("omega"):
            p[n] = uniform(s, 0.5, 2.0)
        else:
            p[n] = uniform(s, -math.pi, math.pi)
    x = normal((c["T"], c["d_in"]), 1.0, tdt) if c["T"] else None
    dy = normal((c["T"], c["d_out"]), 1.0, tdt) if c["kind"] == "step" else None
    return x, dy, p


def _adamw_tensors(c, seed):
    """fp32 parameters, gradients and moments of a layer under training, the
    learning-rate group of each, and bf16 copies of the matrix operands."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    desc = binding.make_desc(1, c["d_in"], c["d_out"], c["r"], "bf16")
    mult = binding.noble_linear_lr_multipliers(desc) if c["r"] else [1.0] * 5
    out = []
    for n in _names(c):
        s = _shape(c, n)
        rn = lambda std: torch.randn(s, generator=g, device="cuda") * std  # noqa: E731
        group = {"W_up": 1, "M": 2}.get(n, 3 if n.startswith("omega") else 4 if n.startswith("phi") else 0)
        t = {"param": rn(0.02), "grad": rn(1e-3), "exp_avg": rn(1e-3), "exp_avg_sq": rn(1e-3).square(),
             "lr_mult": mult[group], "decay": len(s) == 2}
        if n in ("W", "W_down", "W_up"):
            t["param_bf16"] = torch.empty(s, dtype=torch.bfloat16, device="cuda")
        out.append((n, t))
    return out


ADAMW = {"lr": 3e-4, "beta1": 0.9, "beta2": 0.98, "eps": 1e-8, "weight_decay": 0.01, "step": 1000}


def prepare(case, seed):
    c = case
    if c["kind"] == "adamw":
        return {"case": c, "tensors": _adamw_tensors(c, seed)}
    x, dy, p = _tensors(c, seed)
    flags = 0
    if c["r"]:
        flags = binding.NOBLE_FLAG_SIGMA_COS3 if c["sigma"] == "cos3" else binding.SIGMA_FLAGS[c["sigma"]]
    if c["kind"] == "infer":
        flags |= binding.NOBLE_FLAG_INFERENCE
    buf = binding.NobleLinearBuffers(c["T"], c["d_in"], c["d_out"], c["r"], c["dtype"],
                                     with_grads=c["kind"] == "step", flags=flags)
    return {"case": c, "x": x, "dy": dy, "params": p, "buf": buf}


def run(state):
    c = state["case"]
    if c["kind"] == "adamw":
        ts = state["tensors"]
        binding.noble_adamw_step([t for _, t in ts], stream=torch.cuda.current_stream().cuda_stream, **ADAMW)
        return {n: [t["param"], t["exp_avg"], t["exp_avg_sq"], t.get("param_bf16")] for n, t in ts}
    buf, p = state["buf"], state["params"]
    out = {"y": binding.forward(buf, state["x"], p)}
    if c["kind"] == "step":
        out["dx"], grads = binding.backward(buf, state["x"], state["dy"], p)
        out.update({"d" + n: grads["d" + n] for n in _names(c)})
    return out


def work(case):
    c = case
    if c["kind"] == "adamw":
        n = sum(math.prod(_shape(c, k)) for k in _names(c))
        nb = sum(math.prod(_shape(c, k)) for k in _names(c) if k in ("W", "W_down", "W_up"))
        return {"bytes": 28.0 * n + 2.0 * nb, "flops": 0.0}
    T, di, do, es = c["T"], c["d_in"], c["d_out"], 2 if c["dtype"] == "bf16" else 4
    size = {n: math.prod(_shape(c, n)) for n in _names(c)}
    weights = sum(v * (es if n in ("W", "W_down", "W_up") else 4) for n, v in size.items())
    b = es * T * (di + do) + weights
    if c["kind"] == "step":
        b += es * T * (di + do) + 4 * sum(size.values())  # dy in, dx out; fp32 gradients out
    return {"bytes": float(b), "flops": _flops(c)}


def tolerance(case):
    if case["kind"] == "adamw":
        # elementwise fp32 (1e-7); an fp32 step apart, about one bf16 copy in
        # 20000 rounds the other way, 3e-5 of the copies' norm
        return {"rel": 1e-4}
    if case["dtype"] == "fp32":
        # fp32 sums of up to 8192 terms: up to 2e-6 from the 64-bit results
        return {"rel": 1e-5}
    # bf16 outputs (1.7e-3 from the 64-bit results) and a bf16 c, a, db and dh
    # between the contractions (dM 2.3e-3)
    return {"rel": 1e-2}


# ---------------------------------------------------------------- 64-bit results
def _act(sigma):
    """f and f' of a bottleneck without frequencies."""
    if sigma.startswith("tanh"):
        return torch.tanh, lambda u: 1.0 - torch.tanh(u).square()
    if sigma.startswith("leaky"):
        return (lambda u: torch.where(u > 0, u, 0.01 * u)), (lambda u: torch.where(u > 0, 1.0, 0.01).to(u.dtype))
    if sigma.startswith("gelu"):
        cdf = lambda u: 0.5 * (1.0 + torch.erf(u / math.sqrt(2.0)))  # noqa: E731
        pdf = lambda u: torch.exp(-0.5 * u * u) / math.sqrt(2.0 * math.pi)  # noqa: E731
        return (lambda u: u * cdf(u)), (lambda u: cdf(u) + u * pdf(u))
    return (lambda u: u), torch.ones_like


def _exact_adamw(c, seed):
    a, out = ADAMW, {}
    for n, t in _adamw_tensors(c, seed):
        p, g, m, v = (t[k].double() for k in ("param", "grad", "exp_avg", "exp_avg_sq"))
        lr = a["lr"] * t["lr_mult"]
        if t["decay"]:
            p = p - lr * a["weight_decay"] * p
        m = a["beta1"] * m + (1 - a["beta1"]) * g
        v = a["beta2"] * v + (1 - a["beta2"]) * g * g
        den = (v / (1 - a["beta2"] ** a["step"])).sqrt() + a["eps"]
        p = p - lr * (m / (1 - a["beta1"] ** a["step"])) / den
        out[n] = [p, m, v, p.clone() if "param_bf16" in t else None]
    return out


def exact(case, seed):
    c = case
    if c["kind"] == "adamw":
        return _exact_adamw(c, seed)
    x, dy, p = _tensors(c, seed)
    x = x.double()
    p = {n: t.double() for n, t in p.items()}
    s, r, step = c["sigma"], c["r"], c["kind"] == "step"
    y = x @ p["W"].T + p["bias"]
    out = {"y": y}
    layers = []  # (pre-activation, omega, phi) of each layer of the bottleneck
    if r:
        f, df = _act(s)
        pre = x @ p["W_down"].T
        count = {"cos3": 3, "cosnet": 2, "tanh2": 2, "leaky2": 2, "gelu2": 2}.get(s, 1)
        acts = []
        for i in range(count):
            om, ph = p.get("omega%d" % (i + 1)), p.get("phi%d" % (i + 1))
            layers.append(pre)
            acts.append(torch.cos(om * pre + ph) if om is not None else f(pre))
            if i + 1 < count:
                pre = acts[i] @ p["M" if i == 0 else "M2"]
        out["y"] = y + acts[-1] @ p["W_up"].T
    if not step:
        return out
    dy = dy.double()
    out["dx"] = dy @ p["W"]
    out["dW"] = dy.T @ x
    out["dbias"] = dy.sum(0)
    if r:
        out["dW_up"] = dy.T @ acts[-1]
        d = dy @ p["W_up"]
        for i in range(len(layers) - 1, -1, -1):
            u, om, ph = layers[i], p.get("omega%d" % (i + 1)), p.get("phi%d" % (i + 1))
            if om is not None:
                du = -torch.sin(om * u + ph) * d
                out["domega%d" % (i + 1)] = (du * u).sum(0)
                out["dphi%d" % (i + 1)] = du.sum(0)
                d = om * du
            else:
                d = df(u) * d
            if i:
                m = "M" if i == 1 else "M2"
                out["d" + m] = acts[i - 1].T @ d
                d = d @ p[m].T
        out["dW_down"] = d.T @ x
        out["dx"] = out["dx"] + d @ p["W_down"]
    return out
