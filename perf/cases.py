"""Performance cases of the Expert-Token Resonance MoE layer.

A case is one call sequence of the layer's public interface: the forward pass alone ("forward": a layer
that serves or evaluates) or the forward and the backward pass ("step": a layer that trains), on tokens,
parameters and buffers that are on the GPU.  `listed` gives the fixed cases, `draw` more of the same ranges.

Keys of a case: T tokens, d hidden size, D group size of the pooling, E experts, k experts per token, h FFN
hidden size, cf capacity factor, mode "tcr" (token choice) or "ecr" (expert choice), delta_max (the affinity
that fixes the adaptive capacity; 0: the capacity is ceil(cf T k / E)), dtype of the activations, master
(fp32 weights under bf16 activations), gate "affinity" or "softmax", x the distribution of the tokens ("iso":
isotropic, early training; "mix": equally likely clusters, late training; "skew": clusters of very
different weight that lean towards experts, so that a few experts are preferred).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2406_00023_b200 import etr

_BASE = dict(direction="step", D=8, k=2, cf=1.25, mode="tcr", delta_max=0.0, dtype="bf16", master=False,
             gate="affinity", x="iso")


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # A decode step of a serving batch: few tokens, every expert's weights are read for a handful of rows.
        _case("decode_64", direction="forward", T=64, d=1024, E=16, h=2816),
        # The smallest training layer, in fp32 throughout: debugging and reference runs; launches count.
        _case("tiny_f32_step", T=512, d=256, D=4, E=8, h=512, dtype="f32"),
        # An fp32 training step of a batch whose length and widths are no powers of two.
        _case("ragged_f32_step", T=1531, d=768, E=12, h=1000, cf=1.1, dtype="f32", x="mix"),
        # A small model's training step, early (token choice, isotropic tokens, about 512 rows an expert).
        _case("small_step", T=4096, d=1024, E=16, h=2816),
        # A prefill or evaluation pass over a ragged batch.
        _case("prefill_ragged", direction="forward", T=6113, d=2048, E=32, h=1408, x="mix"),
        # Odd sizes everywhere (17 and 23 blocks of 64, 12 experts, three of them per token) and the softmax gate.
        _case("ragged_softmax_step", T=3001, d=1088, E=12, k=3, h=1472, gate="softmax", x="mix"),
        # Many narrow experts with eight of them per token.
        _case("fine_grained_step", T=8192, d=2048, E=128, k=8, h=768, x="mix"),
        # A mid-sized model's step with expert choice: every expert full, late in training.
        _case("mid_ecr_step", T=16384, d=2048, E=32, h=1408, cf=1.0, mode="ecr", x="mix"),
        # Token choice on a skewed load with fp32 master weights (mixed-precision training).
        _case("skew_master_step", T=16384, d=2048, D=16, E=32, h=1408, master=True, x="skew"),
        # Expert choice under an adaptive capacity well below its bound (769 rows of 1280).
        _case("adaptive_ecr_step", T=16384, d=2048, D=16, E=32, h=1408, mode="ecr", delta_max=0.09912, x="skew"),
        # Few wide experts with Top-1 routing: a long prefill.
        _case("top1_prefill", direction="forward", T=32768, d=4096, D=16, E=8, k=1, h=14336, cf=1.0, x="mix"),
        # The largest training step: 64 experts, expert choice, adaptive capacity (about 722 rows of 2048).
        _case("large_step", T=65536, d=4096, D=16, E=64, h=2048, cf=1.0, mode="ecr", delta_max=0.0723, x="mix"),
    ]


def _capacity(c):
    return max(1, int(math.ceil(c["cf"] * c["T"] * c["k"] / c["E"])))


def _rows_per_expert(c):
    """The capacity in use: the bound, or what the adaptive rule makes of delta_max."""
    cap = _capacity(c)
    if c["delta_max"] <= 0.0:
        return cap
    s = c["delta_max"] ** 2
    return max(1, min(cap, int(math.ceil(math.exp(c["d"] * s / (2.0 - s)) / c["E"]))))


def _rows(c):
    """Rows the experts process: full experts in expert choice, k per token within the capacity in token choice."""
    full = c["E"] * min(_rows_per_expert(c), c["T"])
    return full if c["mode"] == "ecr" else min(full, c["T"] * c["k"])


def _flops(c):
    per_row = (6 if c["direction"] == "forward" else 18) * c["d"] * c["h"]
    return per_row * _rows(c) + 2 * c["T"] * c["E"] * (c["d"] // c["D"])


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over their whole ranges on a logarithmic scale, widths in steps of 64 (of 8 in
    fp32), no dearer than the dearest listed one."""
    while True:
        f32 = rng.random() < 0.2
        step = 8 if f32 else 64
        c = _case(direction=rng.choice(["forward", "step", "step"]),
                  T=_log_int(rng, 16, 4096 if f32 else 65536),
                  d=step * _log_int(rng, 256 // step, (1024 if f32 else 4096) // step),
                  h=step * _log_int(rng, 256 // step, (2048 if f32 else 14336) // step),
                  D=rng.choice([4, 8, 16]), E=_log_int(rng, 4, 128), k=rng.choice([1, 2, 2, 3, 4, 8]),
                  cf=rng.choice([1.0, 1.1, 1.25, 1.5]), mode=rng.choice(["tcr", "ecr"]),
                  dtype="f32" if f32 else "bf16", master=not f32 and rng.random() < 0.2,
                  gate=rng.choice(["affinity", "affinity", "affinity", "softmax"]),
                  x=rng.choice(["iso", "mix", "skew"]))
        d, D, E, T = c["d"], c["D"], c["E"], c["T"]
        if d % D or d // D < E or 2 * c["k"] > E:
            continue
        if (E + 35) * (d // D + 8) > 51000:        # the affinity kernels hold all expert embeddings on the chip
            continue
        if rng.random() < 0.25:                    # an adaptive capacity between a third of the bound and the bound
            want = max(1.0, rng.uniform(0.33, 1.0) * _capacity(c))
            y = math.log(want * E)
            c["delta_max"] = round(math.sqrt(2.0 * y / (d + y)), 5)
        weights = 3 * E * d * c["h"] * (4 if f32 or c["master"] else 2) * (2 if c["direction"] == "step" else 1)
        rows = E * (_capacity(c) + 128)
        buffers = rows * (4 * d + 5 * c["h"]) * (4 if f32 else 2) + 4 * T * d * 4
        if weights + buffers > 16e9 or _flops(c) > (8e10 if f32 else 6e12):
            continue
        return c


def _expert_embeddings(E, m, seed):
    """[E, m] fp32 with orthonormal rows."""
    g = np.random.default_rng(seed).standard_normal((m, E))
    q, r = np.linalg.qr(g)
    return torch.from_numpy(np.ascontiguousarray((q * np.sign(np.diag(r))[None, :]).T.astype(np.float32))).cuda()


def _tokens(c, R, gen, dtype):
    """[T, d]: isotropic; or unit-norm cluster means with noise of norm 0.5, in "skew" with means that lean
    towards an expert's direction, Zipf(1.2) weights, and a quarter of the isotropic part left."""
    T, d, E = c["T"], c["d"], c["E"]
    eps = torch.randn(T, d, generator=gen, device="cuda")
    if c["x"] == "iso":
        return eps.to(dtype)
    n = max(8, E)
    mu = torch.nn.functional.normalize(torch.randn(n, d, generator=gen, device="cuda"), dim=1)
    if c["x"] == "mix":
        ids = torch.randint(0, n, (T,), generator=gen, device="cuda")
        alpha, noise = 1.0, 0.5 / math.sqrt(d)
    else:
        lean = R.repeat_interleave(c["D"], dim=1)[torch.arange(n, device="cuda") % E] / math.sqrt(c["D"])
        mu = torch.nn.functional.normalize(0.5 * lean + math.sqrt(0.75) * mu, dim=1)
        p = (torch.arange(n, device="cuda") + 1.0) ** -1.2
        ids = torch.multinomial(p, T, replacement=True, generator=gen)
        alpha = 0.75
        noise = (1.0 - alpha) + alpha * 0.5 / math.sqrt(d)
    return eps.mul_(noise).add_(mu[ids], alpha=alpha).to(dtype)


class _State:
    pass


def _inputs(c, seed):
    """Tokens, expert embeddings, weights and, for a training step, the output's gradient (else None)."""
    act = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    wt = torch.float32 if c["master"] else act
    T, d, E, h = c["T"], c["d"], c["E"], c["h"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    R = _expert_embeddings(E, d // c["D"], seed)
    X = _tokens(c, R, gen, act)

    def weight(*shape):
        w = torch.empty(*shape, dtype=wt, device="cuda")
        for i in range(E):                                   # expert by expert: no second full-size copy
            w[i] = torch.randn(*shape[1:], generator=gen, device="cuda") / math.sqrt(d)
        return w

    W1g, W1u, W2 = weight(E, h, d), weight(E, h, d), weight(E, d, h)
    dY = torch.randn(T, d, generator=gen, device="cuda").to(act) if c["direction"] == "step" else None
    return X, R, W1g, W1u, W2, dY


def prepare(case, seed):
    """Tokens, parameters, gradients and the layer's buffers on the GPU, from the seed alone."""
    c, s = case, _State()
    T, d, E, h = c["T"], c["d"], c["E"], c["h"]
    s.step = c["direction"] == "step"
    s.X, s.R, s.W1g, s.W1u, s.W2, s.dY = _inputs(c, seed)
    s.cfg = etr.make_config(T=T, d=d, D=c["D"], E=E, k=c["k"], h=h, capacity=_capacity(c),
                            dtype=etr.F32 if c["dtype"] == "f32" else etr.BF16,
                            weight_dtype=etr.F32 if s.W2.dtype == torch.float32 else etr.BF16,
                            mode=etr.MODE_ECR if c["mode"] == "ecr" else etr.MODE_TCR,
                            adaptive=c["delta_max"] > 0.0,
                            delta_max_override=c["delta_max"] if c["delta_max"] > 0.0 else -1.0,
                            gate_mode=etr.GATE_SOFTMAX if c["gate"] == "softmax" else etr.GATE_AFFINITY)
    s.buf = etr.LayerBuffers(s.cfg)
    s.Y = torch.empty_like(s.X)
    if s.step:
        s.dX, s.dR = torch.empty_like(s.X), torch.empty_like(s.R)
        s.dW1g, s.dW1u, s.dW2 = torch.empty_like(s.W1g), torch.empty_like(s.W1u), torch.empty_like(s.W2)
    return s


def run(s):
    """One pass: the forward call, and in a training step the backward call."""
    etr.layer_forward(s.cfg, s.X, s.R, s.W1g, s.W1u, s.W2, s.buf, s.Y)
    if not s.step:
        return {"Y": s.Y}
    etr.layer_backward(s.cfg, s.X, s.R, s.W1g, s.W1u, s.W2, s.dY, s.buf, s.dX, s.dR, s.dW1g, s.dW1u, s.dW2)
    return {"Y": s.Y, "dX": s.dX, "dR": s.dR, "dW1g": s.dW1g, "dW1u": s.dW1u, "dW2": s.dW2}


def exact(case, seed):
    """What `run` returns for these inputs, in 64 bits throughout (routing included)."""
    c = case
    T, d, D, E, k = c["T"], c["d"], c["D"], c["E"], c["k"]
    m, C, f64 = d // D, min(_rows_per_expert(c), T), torch.float64
    X, R, W1g, W1u, W2, dY = _inputs(c, seed)
    x, R = X.to(f64), R.to(f64)
    z, a, b = x.view(T, m, D).mean(dim=2), x.norm(dim=1), R.norm(dim=1)
    delta = math.sqrt(D) * (z @ R.T) / (a[:, None] * b[None, :])
    score = delta
    if c["mode"] == "tcr":                     # an expert's candidates: the tokens that have it among their k best
        best = delta.topk(k, dim=1).indices
        score = torch.full_like(delta, -math.inf).scatter_(1, best, delta.gather(1, best))
    gates = torch.softmax(delta, dim=1) if c["gate"] == "softmax" else delta
    rows = []
    for i in range(E):
        val, tok = score[:, i].topk(C)
        rows.append(tok[val > -math.inf].sort().values)

    silu = torch.nn.functional.silu
    Y = torch.zeros(T, d, dtype=f64, device="cuda")
    step = c["direction"] == "step"
    if step:
        dY = dY.to(f64)
        dX, dgate = torch.zeros_like(Y), torch.zeros_like(delta)
        dW = [torch.zeros(w.shape, dtype=f64, device="cuda") for w in (W1g, W1u, W2)]
    for i, t in enumerate(rows):
        wg, wu, w2 = W1g[i].to(f64), W1u[i].to(f64), W2[i].to(f64)
        xp, gt = x[t], gates[t, i][:, None]
        g, u = xp @ wg.T, xp @ wu.T
        hid = silu(g) * u
        o = hid @ w2.T
        Y.index_add_(0, t, gt * o)
        if not step:
            continue
        dgate[t, i] = (dY[t] * o).sum(dim=1)
        do = gt * dY[t]
        dhid, sg = do @ w2, torch.sigmoid(g)
        dg, du = dhid * u * sg * (1.0 + g * (1.0 - sg)), dhid * g * sg
        dX.index_add_(0, t, dg @ wg + du @ wu)
        dW[0][i], dW[1][i], dW[2][i] = dg.T @ xp, du.T @ xp, do.T @ hid
    if not step:
        return {"Y": Y}
    dd = dgate                                 # gradient of the affinities; the selection itself has none
    if c["gate"] == "softmax":
        dd = gates * (dgate - (gates * dgate).sum(dim=1, keepdim=True))
    w = dd * math.sqrt(D) / (a[:, None] * b[None, :])
    dX += ((w @ R) / D).repeat_interleave(D, dim=1) - ((dd * delta).sum(dim=1) / a ** 2)[:, None] * x
    dR = w.T @ z - ((dd * delta).sum(dim=0) / b ** 2)[:, None] * R
    return {"Y": Y, "dX": dX, "dR": dR, "dW1g": dW[0], "dW1u": dW[1], "dW2": dW[2]}


def work(case):
    """Inputs read once, outputs written once, and the arithmetic of the rows the experts process; an expert
    without a row (few tokens) needs no weights."""
    c = case
    T, d, E, h, m = c["T"], c["d"], c["E"], c["h"], c["d"] // c["D"]
    b = 4 if c["dtype"] == "f32" else 2
    wb = 4 if c["master"] else b
    in_use = E * (1.0 - (1.0 - min(1.0, c["k"] / E)) ** T) if c["mode"] == "tcr" else E
    weights = 3.0 * d * h * wb
    if c["direction"] == "forward":
        nbytes = 2 * T * d * b + E * m * 4 + in_use * weights
    else:
        nbytes = 4 * T * d * b + 2 * E * m * 4 + in_use * weights + E * weights
    return {"bytes": nbytes, "flops": float(_flops(c))}


def tolerance(case):
    """About four times what the layer shows against itself in 64 bits on the same routing (relative 2-norm, the
    worst output of each case): bf16 2.9e-3 to 3.7e-3 (three to five roundings to bf16 on the way to an
    output), fp32 8e-7 to 1.2e-6."""
    return {"rel": 1.2e-2} if case["dtype"] == "bf16" else {"rel": 5e-6}
