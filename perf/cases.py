"""The work that users of this library have it do, as cases to be timed.

A case is a dict of plain values: ``kind`` says which public entry points a pass goes through, the rest are
sizes and options.  ``prepare`` makes what a training program holds before the call (activations, output
cotangents, parameters, optimizer state, buffers it keeps), ``run`` is one pass of the calls such a program makes.
Activations are N(0,1) (what a normalisation layer hands on), cotangents are Student-t(3) or Gaussian with a
tenth of the examples scaled up, as in ``inputs``; B is the number of examples, T the tokens of each.
"""
import math

import torch

import paper_2510_00236_b200 as pe
from paper_2510_00236_b200 import conv_unfold, inputs

DEV = "cuda:0"
BF16 = torch.bfloat16
ADAM = dict(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8)
SIGN = dict(lr=3.47e-3, beta=0.9)
# from this many input elements on, the two-pass form of the per-token statistic is the one to call
TOKEN_STAGED_MIN_ELEMS = 100_000_000


def listed():
    return [
        # One small fp32 layer, every statistic and a MicroAdam step: the smallest calls, where latency counts.
        dict(name="fp32_small", kind="fp32", B=8, T=16, d_in=64, d_out=64),
        # The same calls on an ordinary fp32 layer (full-precision training of a small model).
        dict(name="fp32_layer", kind="fp32", B=32, T=128, d_in=256, d_out=1024),
        # A training step's statistics and MicroAdam updates over all 25 linear layers of a 6-layer decoder.
        dict(name="decoder_step", kind="decoder", B=64, T=256, layers=6, d_model=512, d_mlp=2048, vocab=32768),
        # An MLP layer of a small transformer: mean, square and sign, the per-token statistic, both optimizer steps.
        dict(name="mlp_step", kind="step", B=64, T=256, d_in=512, d_out=2048),
        # The same for the large layer: the largest single-GPU work.
        dict(name="large_step", kind="step", B=256, T=1024, d_in=2048, d_out=8192),
        # Many short sequences (sentence classification, reward models): mean and square.
        dict(name="short_square", kind="short", what="square", B=1024, T=32, d_in=1024, d_out=1024),
        # Short sequences through a wide layer: mean, square and sign in one pass.
        dict(name="short_all", kind="short", what="all", B=128, T=32, d_in=4096, d_out=4096),
        # A packed batch of unequal lengths (instruction tuning), then MicroAdam.
        dict(name="packed", kind="packed", B=96, mean_len=300, d_in=512, d_out=2048),
        # Per-example clipping with one norm over an MLP's two layers (private training).
        dict(name="clipped", kind="clipped", B=64, T=256, d_in=512, d_out=2048),
        # Statistics and MicroAdam in one call without statistic buffers (memory-bound training).
        dict(name="lean_step", kind="lean", B=32, T=512, d_in=1024, d_out=4096),
        # The unembedding of a vocabulary whose size is no multiple of 8.
        dict(name="unembed_odd", kind="odd", B=8, T=256, d_in=1024, d_out=32101),
        # The first convolution of an image model through the unfolded contraction.
        dict(name="conv_first", kind="conv", B=32, C=3, size=112, K=7, stride=2, F=64),
    ]


def _log_int(rng, lo, hi, multiple=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))
    return min(hi, max(lo, int(v) // multiple * multiple))


def draw(rng):
    """One more case: the kinds of listed() over the sizes they stand for."""
    kind = rng.choice(["fp32", "decoder", "step", "short", "short", "packed", "clipped", "lean", "odd", "conv"])
    while True:
        if kind == "fp32":
            c = dict(B=_log_int(rng, 4, 64), T=_log_int(rng, 8, 256), d_in=_log_int(rng, 48, 1100), d_out=_log_int(rng, 48, 1100))
            ok = c["B"] * c["T"] * c["d_in"] * c["d_out"] <= 2 ** 31
        elif kind == "decoder":
            d = 64 * rng.randint(2, 10)
            c = dict(B=_log_int(rng, 16, 96), T=_log_int(rng, 64, 512), layers=rng.randint(2, 6), d_model=d, d_mlp=4 * d, vocab=8 * _log_int(rng, 500, 4096))
            ok = c["B"] * c["T"] <= 20000
        elif kind == "step":
            c = dict(B=_log_int(rng, 16, 256), T=_log_int(rng, 64, 1024), d_in=_log_int(rng, 256, 4096, 8), d_out=_log_int(rng, 256, 8192, 8))
            ok = 2 ** 32 <= c["B"] * c["T"] * c["d_in"] * c["d_out"] <= 2 ** 41
        elif kind == "short":
            c = dict(what=rng.choice(["square", "sign", "all"]), B=_log_int(rng, 64, 2048), T=_log_int(rng, 1, 32),
                     d_in=_log_int(rng, 256, 4096, 8), d_out=_log_int(rng, 256, 4096, 8))
            ok = c["B"] * c["d_in"] * c["d_out"] <= 2 ** 33
        elif kind == "packed":
            c = dict(B=_log_int(rng, 16, 256), mean_len=_log_int(rng, 30, 800), d_in=_log_int(rng, 256, 2048, 8), d_out=_log_int(rng, 256, 4096, 8))
            ok = c["B"] * c["mean_len"] * c["d_in"] * c["d_out"] <= 2 ** 38
        elif kind == "clipped":
            c = dict(B=_log_int(rng, 16, 256), T=_log_int(rng, 32, 512), d_in=_log_int(rng, 256, 2048, 8), d_out=_log_int(rng, 256, 4096, 8))
            ok = c["B"] * c["T"] * c["d_in"] * c["d_out"] <= 2 ** 38
        elif kind == "lean":
            c = dict(B=_log_int(rng, 16, 128), T=_log_int(rng, 64, 1024), d_in=_log_int(rng, 512, 2048, 8), d_out=_log_int(rng, 512, 8192, 8))
            ok = c["B"] * c["T"] * c["d_in"] * c["d_out"] <= 2 ** 38
        elif kind == "odd":
            c = dict(B=_log_int(rng, 4, 32), T=_log_int(rng, 32, 512), d_in=_log_int(rng, 256, 1200), d_out=_log_int(rng, 1000, 33000))
            ok = (c["d_in"] % 8 or c["d_out"] % 8) and 2 ** 30 <= c["B"] * c["T"] * c["d_in"] * c["d_out"] <= 2 ** 36
        else:
            c = dict(B=_log_int(rng, 8, 64), C=rng.choice([1, 3, 4, 16, 64]), size=rng.randint(14, 112), K=rng.choice([3, 5, 7]), stride=rng.choice([1, 2]), F=rng.choice([32, 48, 64, 96, 128]))
            t = ((c["size"] - 1) // c["stride"] + 1) ** 2
            ok = c["B"] * t * c["C"] * c["K"] ** 2 <= 60_000_000
        if ok:
            return dict(kind=kind, **c)


def _decoder_layers(c):
    """(d_in, d_out) of every linear layer: fused QKV, output projection, MLP up and down per block, unembedding."""
    d, m = c["d_model"], c["d_mlp"]
    return [(d, 3 * d), (d, d), (d, m), (m, d)] * c["layers"] + [(d, c["vocab"])]


def _layer(c, seed, T=None, d_in=None, d_out=None, dtype=BF16):
    """X ~ N(0,1), dY ~ N(0,1/T) with a seeded tenth of the examples times 5."""
    B, T, d_in, d_out = c["B"], T or c["T"], d_in or c["d_in"], d_out or c["d_out"]
    g = torch.Generator(device=DEV).manual_seed(seed)
    X = torch.randn((B, T, d_in), generator=g, device=DEV, dtype=torch.float32 if dtype == torch.float32 else BF16).to(dtype)
    dY = torch.randn((B, T, d_out), generator=g, device=DEV, dtype=torch.float32 if dtype == torch.float32 else BF16)
    boost = 1.0 + 4.0 * (torch.rand((B, 1, 1), generator=g, device=DEV) < 0.1).float()
    return X, dY.mul_((boost * T ** -0.5).to(dY.dtype)).to(dtype)


def _params(d_in, d_out, seed, low_precision=True):
    """fp32 master weights, MicroAdam's two moments, and the bf16 copy the next forward pass reads."""
    theta = inputs.master_weights(d_out, d_in, seed, DEV)
    p = dict(theta=theta, m=torch.zeros_like(theta), v=torch.zeros_like(theta))
    if low_precision:
        p["lp"] = theta.to(BF16)
    return p


def _new(d_in, d_out):
    return torch.empty((d_out, d_in), dtype=torch.float32, device=DEV)


def prepare(case, seed):
    c, s = case, dict(case=case, step=0)
    kind = c["kind"]
    if kind == "fp32":
        s["X"], s["dY"] = _layer(c, seed, dtype=torch.float32)
        s["p"] = _params(c["d_in"], c["d_out"], seed + 1, low_precision=False)
    elif kind == "decoder":
        s["layers"] = []
        for k, (d_in, d_out) in enumerate(_decoder_layers(c)):
            X, dY = _layer(c, seed + 97 * k, d_in=d_in, d_out=d_out)
            if d_in == c["d_mlp"]:
                X = torch.nn.functional.gelu(X)         # what the MLP's down projection is given
            s["layers"].append(dict(X=X, dY=dY, mean=_new(d_in, d_out), stat=_new(d_in, d_out), p=_params(d_in, d_out, seed + k)))
    elif kind == "step":
        li = inputs.heavy_tailed_layer(c["B"], c["T"], c["d_in"], c["d_out"], seed=seed, device=DEV, with_weights=False)
        s["X"], s["dY"] = li.X, li.dY
        s["p"] = _params(c["d_in"], c["d_out"], seed + 1)
        s["q"] = _params(c["d_in"], c["d_out"], seed + 2)
        s["out"] = [_new(c["d_in"], c["d_out"]) for _ in range(4)]
        s["staged"] = c["B"] * c["T"] * (c["d_in"] + c["d_out"]) >= TOKEN_STAGED_MIN_ELEMS
        if s["staged"]:
            need = pe.pe_token_sqstats_staged_workspace_bytes(c["B"], c["T"], c["d_in"], c["d_out"])
            s["ws"] = torch.empty(max(need, 1), dtype=torch.uint8, device=DEV)
    elif kind == "packed":
        g = torch.Generator().manual_seed(seed)
        lens = (c["mean_len"] * torch.exp(0.6 * torch.randn(c["B"], generator=g) - 0.18)).long().clamp(1, 4 * c["mean_len"])
        offs = torch.cat([torch.zeros(1, dtype=torch.long), lens.cumsum(0)])
        s["offs"] = offs.to(torch.int32).to(DEV)
        X, dY = _layer(dict(B=1), seed, T=int(offs[-1]), d_in=c["d_in"], d_out=c["d_out"])
        s["X"], s["dY"] = X[0], dY[0].mul_(math.sqrt(c["B"]))        # per sequence ~ N(0, 1 / mean length)
        s["mean"], s["stat"] = _new(c["d_in"], c["d_out"]), _new(c["d_in"], c["d_out"])
        need = pe.pe_linear_stats_ragged_workspace_bytes(c["B"], c["d_in"], c["d_out"])
        s["ws"] = torch.empty(max(need, 1), dtype=torch.uint8, device=DEV)
        s["p"] = _params(c["d_in"], c["d_out"], seed + 1)
    elif kind == "clipped":
        X, dY = _layer(c, seed)
        X2, dY2 = _layer(c, seed + 97, d_in=c["d_out"], d_out=c["d_in"])
        s["layers"] = [(X, dY), (torch.nn.functional.gelu(X2), dY2)]
        # a norm bound near the typical example's, so that some are clipped and some are not
        s["clip"] = math.sqrt(1.45 * c["d_in"] * c["d_out"])
    elif kind == "lean":
        s["X"], s["dY"] = _layer(c, seed)
        s["p"] = _params(c["d_in"], c["d_out"], seed + 1)
    elif kind == "conv":
        g = torch.Generator(device=DEV).manual_seed(seed)
        out = (c["size"] - 1) // c["stride"] + 1
        s["x"] = torch.randn((c["B"], c["C"], c["size"], c["size"]), generator=g, device=DEV).to(BF16)
        s["gy"] = (torch.randn((c["B"], c["F"], out, out), generator=g, device=DEV) / out).to(BF16)
    else:
        s["X"], s["dY"] = _layer(c, seed)
    return s


def _microadam(s, p, mean, stat):
    pe.microadam_step(p["theta"], p["m"], p["v"], mean, stat, s["case"]["B"], step=s["step"], theta_lp=p.get("lp"), **ADAM)


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    s["step"] += 1
    if kind == "fp32":
        mean, square = pe.pe_linear_stats_f32(s["X"], s["dY"], "square")
        _, sign = pe.pe_linear_stats_f32(s["X"], s["dY"], "sign", None, torch.empty_like(mean))
        token = pe.pe_token_sqstats_f32(s["X"], s["dY"])
        _microadam(s, s["p"], mean, square)
        return mean, square, sign, token, s["p"]
    if kind == "decoder":
        out = []
        for layer in s["layers"]:
            pe.pe_linear_stats(layer["X"], layer["dY"], "square", layer["mean"], layer["stat"])
            _microadam(s, layer["p"], layer["mean"], layer["stat"])
            out.append((layer["mean"], layer["stat"]))
        # 64 outputs at most are compared: every layer's statistics, and the parameters of the first three and the last
        return out[:24] + out[-1:], [layer["p"]["theta"] for layer in s["layers"][:3] + s["layers"][-1:]]
    if kind == "step":
        mean, square, sign, token = s["out"]
        pe.pe_linear_stats_all(s["X"], s["dY"], mean, square, sign)
        if s["staged"]:
            pe.pe_token_sqstats_staged(s["X"], s["dY"], token, s["ws"])
        else:
            pe.pe_token_sqstats(s["X"], s["dY"], token)
        _microadam(s, s["p"], mean, square)
        pe.microsignsgd_step(s["q"]["theta"], s["q"]["m"], sign, c["B"], theta_lp=s["q"]["lp"], **SIGN)
        return mean, square, sign, token, s["p"], s["q"]["theta"], s["q"]["m"], s["q"]["lp"]
    if kind == "short":
        if c["what"] == "all":
            return pe.pe_linear_stats_all(s["X"], s["dY"])
        if c["what"] == "sign":
            return pe.pe_linear_stats(s["X"], s["dY"], "sign", None, _new(c["d_in"], c["d_out"]))
        return pe.pe_linear_stats(s["X"], s["dY"], "square")
    if kind == "packed":
        pe.pe_linear_stats_ragged(s["X"], s["dY"], s["offs"], "square", s["mean"], s["stat"], s["ws"])
        _microadam(s, s["p"], s["mean"], s["stat"])
        return s["mean"], s["stat"], s["p"]
    if kind == "clipped":
        norms = [pe.pe_example_sqnorms(X, dY) for X, dY in s["layers"]]
        total = norms[0] + norms[1]
        return total, [pe.pe_linear_clipped_sum(X, dY, s["clip"], total)[0] for X, dY in s["layers"]]
    if kind == "lean":
        p = s["p"]
        pe.pe_linear_microadam_step(s["X"], s["dY"], p["theta"], p["m"], p["v"], step=s["step"], theta_lp=p["lp"], **ADAM)
        return p
    if kind == "conv":
        return conv_unfold.pe_conv2d_stats(s["x"], s["gy"], (c["F"], c["C"], c["K"], c["K"]), "square", c["stride"], c["K"] // 2)
    return pe.pe_linear_stats(s["X"], s["dY"], "square")


def work(case):
    """One pass: inputs read once, results written once, parameters and moments read and written once."""
    c, kind = case, case["kind"]

    def layer(rows, d_in, d_out, outs, in_bytes=2):
        return rows * (d_in + d_out) * in_bytes + 4 * outs * d_in * d_out, 2 * rows * d_in * d_out

    adam = lambda n, lp=2: (24 + lp) * n         # noqa: E731  theta, m, v in and out, the bf16 copy out
    b = f = 0
    if kind == "fp32":
        b, f = layer(c["B"] * c["T"], c["d_in"], c["d_out"], 4, 4)
        b, f = b + adam(c["d_in"] * c["d_out"], 0), 2 * f        # the per-example and the per-token contraction
    elif kind == "decoder":
        for d_in, d_out in _decoder_layers(c):
            lb, lf = layer(c["B"] * c["T"], d_in, d_out, 2)
            b, f = b + lb + adam(d_in * d_out), f + lf
    elif kind == "step":
        b, f = layer(c["B"] * c["T"], c["d_in"], c["d_out"], 4)
        b, f = b + (26 + 18) * c["d_in"] * c["d_out"], 2 * f
    elif kind == "short":
        b, f = layer(c["B"] * c["T"], c["d_in"], c["d_out"], {"square": 2, "sign": 1, "all": 3}[c["what"]])
    elif kind == "packed":
        b, f = layer(c["B"] * c["mean_len"], c["d_in"], c["d_out"], 2)
        b += adam(c["d_in"] * c["d_out"])
    elif kind == "clipped":
        b, f = layer(c["B"] * c["T"], c["d_in"], c["d_out"], 1)
        b, f = 2 * b, 2 * f
    elif kind == "lean":
        b, f = layer(c["B"] * c["T"], c["d_in"], c["d_out"], 0)
        b += adam(c["d_in"] * c["d_out"])
    elif kind == "conv":
        out = (c["size"] - 1) // c["stride"] + 1
        d_in = c["C"] * c["K"] ** 2
        b = 2 * c["B"] * (c["C"] * c["size"] ** 2 + c["F"] * out * out) + 8 * d_in * c["F"]
        f = 2 * c["B"] * out * out * d_in * c["F"]
    else:
        b, f = layer(c["B"] * c["T"], c["d_in"], c["d_out"], 2)
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times the largest difference from the same pass in 64 bits, over listed and drawn cases.

    Sums of fp32 products: 1.1e-6 (2-norm), 5e-6 (largest entry).  MicroAdam's v: 1.5e-5, from 1 - beta2 in fp32.
    The bf16 parameter copy: an entry on a rounding boundary moves by 2^-8.  Sign sums: an entry of G_b within
    rounding of zero may count as the other sign, a change of 2 where the sums are about sqrt(B)."""
    if case["kind"] in ("fp32", "step"):
        return {"rel": 4e-3, "max": 0.9}
    if case["kind"] == "short":
        return {"rel": 1e-5, "max": 4e-5} if case["what"] == "square" else {"rel": 3e-4, "max": 0.9}
    if case["kind"] in ("decoder", "packed", "lean"):
        return {"rel": 6e-5, "max": 0.02}
    return {"rel": 1e-5, "max": 4e-5}
