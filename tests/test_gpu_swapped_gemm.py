"""The bf16 grouped GEMMs with the weights as the M operand and the tokens as N, stage by stage: row counts around
the 16-row steps and the 256-row tiles, column counts that end inside a tile, every size of token box, all four
epilogues, against 64-bit products of the same bf16 inputs, and bit for bit against the CTA-pair form; beside them the
weight gradients (one launch of their own in both) against the same products and bit for bit against the single-CTA form, in
bf16 and in fp32, whose buffers start as NaN: experts without rows included.

Tolerance (relative 2-norm): an output is one rounding to bf16, at most 2^-8 of a value and 1.66e-3 in the root mean
square; the fp32 sums are three orders below.  2.5e-3 leaves room for small blocks, whose rms scatters.  fp32 gradients
are those sums: at most 600 products, whose accumulator cuts 2^-24 of the sum on average at each of 38 MMAs: 1e-6 leaves
room for the cuts all pointing one way."""
import math

import pytest
import torch

from paper_2406_00023_b200 import etr

pytestmark = pytest.mark.gpu
TOL = 2.5e-3


def rel(got, ref):
    n = float(ref.norm())
    return float((got.double() - ref).norm()) / n if n else float(got.double().norm())


def run(E, d, h, cap, counts, impl, grad_fp32=False, wait_limit_cycles=0):
    g = torch.Generator(device="cuda").manual_seed(1)
    cfg = etr.make_config(T=max(8, cap), d=d, D=1, E=E, k=1, h=h, capacity=cap, dtype=etr.BF16, mode=etr.MODE_TCR,
                          gemm_impl=impl, grad_fp32=grad_fp32, wait_limit_cycles=wait_limit_cycles)
    assert etr.validate(cfg) == etr.OK
    b = etr.LayerBuffers(cfg)
    b.block.fill_(0xFF)                                      # NaN wherever nothing is written
    b.stats.zero_()
    b.counts.copy_(torch.tensor(counts, dtype=torch.int32))
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    W = [(rnd(*s) / math.sqrt(d)).bfloat16() for s in ((E, h, d), (E, h, d), (E, d, h))]
    Cs = etr.c_stride(cfg)
    for t in (b.Xp, b.dO):
        v = t.view(E, Cs, d)
        for i, n in enumerate(counts):
            v[i, :n] = rnd(n, d).bfloat16()
            v[i, n:(n + 127) // 128 * 128] = 0.0
    dW = [torch.full_like(w, float("nan"), dtype=torch.float32 if grad_fp32 else None) for w in W]
    etr.expert_ffn(cfg, b.route, b.Xp, *W, b.G, b.U, b.H, b.O, b.c.stats, b.c.ws)
    etr.expert_ffn_bwd(cfg, b.route, b.dO, b.Xp, b.G, b.U, b.H, *W, b.dG, b.dU, b.dXp, *dW, b.c.stats, b.c.ws)
    assert b.read_stats().error_word == 0
    return b, W, Cs, dW


@pytest.mark.parametrize("E,d,h,cap,counts", [
    (4, 64, 64, 10, (10, 0, 1, 7)),                          # boxes of 8 rows, one tile of 16
    (3, 128, 192, 32, (32, 17, 16)),                         # boxes of 16
    (3, 320, 448, 64, (64, 33, 49)),                         # boxes of 32, column tiles end inside
    (5, 256, 320, 192, (192, 129, 128, 127, 15)),            # boxes of 64
    (9, 4096, 256, 600, (600, 512, 513, 511, 257, 256, 255, 0, 1)),      # two and three tiles per expert
    (38, 1600, 128, 300, tuple((53 * i) % 301 for i in range(38))),      # many tiles, plain stores only
])
def test_stages(E, d, h, cap, counts):
    b, W, Cs, dW = run(E, d, h, cap, counts, etr.GEMM_AUTO)
    p, *_ = run(E, d, h, cap, counts, etr.GEMM_TCGEN05_2CTA)
    *_, dWs = run(E, d, h, cap, counts, etr.GEMM_TCGEN05)
    f, _, _, dWf = run(E, d, h, cap, counts, etr.GEMM_AUTO, grad_fp32=True)
    assert all(torch.equal(u, v) for u, v in zip(dW, dWs)) and all(torch.equal(u, v.bfloat16()) for u, v in zip(dW, dWf))
    for i, n in enumerate(counts):
        pad = (n + 127) // 128 * 128
        x, G, U, H, O, dO, dG, dU, dXp = (t.view(E, Cs, -1)[i].double() for t in
                                          (b.Xp, b.G, b.U, b.H, b.O, b.dO, b.dG, b.dU, b.dXp))
        for t in (G, U, H, O, dG, dU, dXp):
            assert bool((t[n:pad] == 0).all()) and bool(t[pad:].isnan().all())
        if n == 0:
            assert all(bool((t[i] == 0).all()) for t in (*dW, *dWf))
            continue
        x, G, U, H, O, dO, dG, dU, dXp = (t[:n] for t in (x, G, U, H, O, dO, dG, dU, dXp))
        wg, wu, w2 = (w[i].double() for w in W)
        g32, u32, s, dh = x @ wg.T, x @ wu.T, torch.sigmoid(G), dO @ w2
        for name, got, ref in (("G", G, g32), ("U", U, u32), ("H", H, torch.nn.functional.silu(g32) * u32),
                               ("O", O, H @ w2.T), ("dG", dG, dh * U * s * (1 + G * (1 - s))), ("dU", dU, dh * G * s),
                               ("dXp", dXp, dG @ wg + dU @ wu)):
            assert rel(got, ref) <= TOL, (name, i, rel(got, ref))
            assert torch.equal(got, getattr(p, name).view(E, Cs, -1)[i][:n].double()), (name, i)
        for name, got, g32, ref in (("dW1g", dW[0], dWf[0], dG.T @ x), ("dW1u", dW[1], dWf[1], dU.T @ x), ("dW2", dW[2], dWf[2], dO.T @ H)):
            assert rel(got[i], ref) <= TOL and rel(g32[i], ref) <= 1e-6, (name, i, rel(got[i], ref), rel(g32[i], ref))
