"""The fp32 grouped GEMMs on the tensor cores, stage by stage against 64-bit products of the same inputs: sizes at
the edges of the 128-row and 128- or 64-column tiles and of the 32-wide K blocks, row counts from none to a full
buffer, and values at the ends of the number range.

Tolerance (relative 2-norm): a value split into two tf32 parts is off by at most 2^-23, the dropped lo*lo by 2^-22 of
a product at most, and a chain of four MMAs drops at most four last bits of its sum (2^-23 each): 1e-6 holds all
of it with the growth of the running sum's roundings over the K blocks (2^-24 sqrt(K / 32) at K <= 2000)."""
import math

import numpy as np
import pytest
import torch

from gen import workloads as gw
from oracle import binding as ob
from paper_2406_00023_b200 import etr
from tests import harness as hz

pytestmark = pytest.mark.gpu
TOL = 1e-6


def rel(got, ref):
    n = float(ref.norm())
    return float((got.double() - ref).norm()) / n if n else float(got.double().norm())


def layer(E, d, h, cap, counts, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    cfg = etr.make_config(T=max(8, cap), d=d, D=1, E=E, k=1, h=h, capacity=cap, dtype=etr.F32, mode=etr.MODE_TCR)
    assert etr.validate(cfg) == etr.OK
    b = etr.LayerBuffers(cfg)
    b.block.fill_(0xFF)                                      # NaN wherever nothing is written
    b.stats.zero_()
    b.counts.copy_(torch.tensor(counts, dtype=torch.int32))
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    W = [rnd(E, h, d) / math.sqrt(d), rnd(E, h, d) / math.sqrt(d), rnd(E, d, h) / math.sqrt(d)]
    Cs = etr.c_stride(cfg)
    for t in (b.Xp, b.dO):
        v = t.view(E, Cs, d)
        for i, n in enumerate(counts):
            v[i, :n] = rnd(n, d)
            v[i, n:(n + 127) // 128 * 128] = 0.0
    return cfg, b, W


@pytest.mark.parametrize("E,d,h,cap,counts", [
    (3, 8, 8, 5, (5, 0, 1)),                                 # one partial K block, one partial tile
    (4, 40, 72, 129, (129, 128, 127, 0)),                    # K blocks and column tiles end inside
    (5, 256, 1000, 300, (300, 33, 1, 256, 65)),              # several row tiles, 64- and 128-column tiles
    (2, 1096, 136, 700, (700, 641)),
    (24, 512, 768, 257, tuple((37 * i) % 258 for i in range(24))),       # more tiles than SMs
])
def test_stages_against_64_bits(E, d, h, cap, counts):
    cfg, b, W = layer(E, d, h, cap, counts)
    dW = [torch.full_like(w, float("nan")) for w in W]
    etr.expert_ffn(cfg, b.route, b.Xp, *W, b.G, b.U, b.H, b.O, b.c.stats, b.c.ws)
    etr.expert_ffn_bwd(cfg, b.route, b.dO, b.Xp, b.G, b.U, b.H, *W, b.dG, b.dU, b.dXp, *dW, b.c.stats, b.c.ws)
    assert b.read_stats().error_word == 0
    Cs = etr.c_stride(cfg)
    for i, n in enumerate(counts):
        pad = (n + 127) // 128 * 128
        x, G, U, H, O, dO, dG, dU, dXp = (t.view(E, Cs, -1)[i].double() for t in
                                          (b.Xp, b.G, b.U, b.H, b.O, b.dO, b.dG, b.dU, b.dXp))
        for t in (G, U, H, O, dG, dU, dXp):
            assert bool((t[n:pad] == 0).all()) and bool(t[pad:].isnan().all())
        x, G, U, H, O, dO, dG, dU, dXp = (t[:n] for t in (x, G, U, H, O, dO, dG, dU, dXp))
        wg, wu, w2 = (w[i].double() for w in W)
        s, dh = torch.sigmoid(G), dO @ w2
        for name, got, ref in (("G", G, x @ wg.T), ("U", U, x @ wu.T), ("H", H, G * s * U), ("O", O, H @ w2.T),
                               ("dG", dG, dh * U * s * (1 + G * (1 - s))), ("dU", dU, dh * G * s),
                               ("dXp", dXp, dG @ wg + dU @ wu), ("dW1g", dW[0][i], dG.T @ x),
                               ("dW1u", dW[1][i], dU.T @ x), ("dW2", dW[2][i], dO.T @ H)):
            assert rel(got, ref) <= TOL, (name, i, rel(got, ref))


@pytest.mark.parametrize("d", [64, 512])                      # chains of two and of four MMAs
def test_ends_of_the_number_range(d):
    """An infinity gives the infinities that fp32 products give, a NaN its row, the largest and the smallest finite
    values their products; the other rows of the tile are as if these were not there."""
    cfg, b, W = layer(1, d, 64, 128, (128,))
    x = b.Xp.view(128, d)
    x[3, 7], x[4, 9], x[5, 63] = math.inf, -math.inf, math.nan
    x[6] = 0.0
    x[6, 1] = torch.finfo(torch.float32).max
    x[7] = 0.0
    x[7, 2] = 1e-30
    etr.expert_ffn(cfg, b.route, b.Xp, *W, b.G, b.U, b.H, b.O, b.c.stats, b.c.ws)
    assert b.read_stats().error_word == 0
    ref = x.double() @ W[0][0].double().T
    G = b.G.view(128, 64).double()
    for r in (3, 4):
        assert bool((G[r] == ref[r]).all())                  # +-inf by the weight's sign
    assert bool(G[5].isnan().all())
    for r in (6, 7):
        ok = ref[r].abs() < 3e38
        assert bool((G[r][ok] - ref[r][ok]).abs().le(1e-6 * ref[r][ok].abs()).all())
    rest = [r for r in range(128) if r not in (3, 4, 5, 6, 7)]
    assert rel(G[rest], ref[rest]) <= TOL


@pytest.mark.parametrize("exponent", [-100, -112, -116, -120, -124])
def test_small_values_lose_the_bits_below_the_tf32_range(exponent):
    """The smallest step of a tf32 value is 2^-136, so that lo is off by up to 2^-137 whatever the size of the value: below
    the format's own error down to values of 2^-113, and 2^-137 of the value's size beyond."""
    cfg, b, W = layer(1, 64, 64, 128, (128,))
    b.Xp.view(128, 64).mul_(2.0 ** exponent)
    etr.expert_ffn(cfg, b.route, b.Xp, *W, b.G, b.U, b.H, b.O, b.c.stats, b.c.ws)
    ref = b.Xp.view(128, 64).double() @ W[0][0].double().T
    assert rel(b.G.view(128, 64), ref) <= 2e-7 + 2.0 ** (-137 - exponent)


@pytest.mark.parametrize("d", [64, 512])
@pytest.mark.parametrize("bits", [0x7f800001, 0x7f801fff, -0x7fffff, -0x7fe001, 0x7fc00000, -1])
def test_every_nan_stays_a_nan(bits, d):
    """Payloads in the low 13 bits only (0x7f800001, 0x7f801fff and the negative ones), the canonical NaN and all ones,
    in a token, a weight and a gradient: NaN in exactly the outputs whose products hold it."""
    cfg, b, W = layer(1, d, 64, 128, (128,))
    put = lambda t, *at: t.view(torch.int32).__setitem__(at, bits)  # noqa: E731
    x, dO = b.Xp.view(128, d), b.dO.view(128, d)
    put(x, 3, 7)
    put(W[1], 0, 5, 9)
    put(dO, 11, 2)
    dW = [torch.empty_like(w) for w in W]
    etr.expert_ffn(cfg, b.route, b.Xp, *W, b.G, b.U, b.H, b.O, b.c.stats, b.c.ws)
    etr.expert_ffn_bwd(cfg, b.route, b.dO, b.Xp, b.G, b.U, b.H, *W, b.dG, b.dU, b.dXp, *dW, b.c.stats, b.c.ws)
    assert b.read_stats().error_word == 0
    G, U, dG = (t.view(128, 64).isnan() for t in (b.G, b.U, b.dG))
    row, col = torch.arange(128, device="cuda")[:, None], torch.arange(64, device="cuda")[None, :]
    assert G.equal((row == 3).expand(128, 64)) and U.equal((row == 3) | (col == 5))
    assert dG.equal((row == 3) | (row == 11) | (col == 5))
    assert bool(dW[2].isnan()[0, 2].all())                   # its row of dO, transposed on the way


@pytest.mark.parametrize("d,h,n", [(64, 392, 256), (256, 64, 250), (384, 256, 48), (128, 128, 64)])
def test_short_contractions_are_cut_less(d, h, n):
    """Positive operands, so that every cut of the accumulator counts: half a last bit of a sum whose mantissa is 1.44 on
    average, 2^-24 / 1.44 = 4.1e-8, at each MMA for the part of the chain summed so far: 1.5 times that for two MMAs, 2.5
    times for four.  Beside it, independent: a rounding of the running sum per chain, 2^-24 / sqrt(3) / 1.2 of the part
    summed so far (root mean square of the parts: 1 / sqrt(3)), and the operands' (3e-8 in all).  A tenth on top."""
    def bound(k):
        mmas = 2 if k <= 384 else 4
        cut = (1 + mmas) / 2 * 2.0 ** -24 / 1.44
        return 1.1 * math.sqrt(cut ** 2 + k / (8 * mmas) / 3 * (2.0 ** -24 / 1.2 / math.sqrt(3)) ** 2 + 3e-8 ** 2)

    cfg, b, W = layer(2, d, h, n, (n, n))
    Cs = etr.c_stride(cfg)
    for t in (b.Xp, b.dO):
        t.view(2, Cs, d)[:, :n].abs_()
    for w in W:
        w.abs_()
    dW = [torch.empty_like(w) for w in W]
    etr.expert_ffn(cfg, b.route, b.Xp, *W, b.G, b.U, b.H, b.O, b.c.stats, b.c.ws)
    etr.expert_ffn_bwd(cfg, b.route, b.dO, b.Xp, b.G, b.U, b.H, *W, b.dG, b.dU, b.dXp, *dW, b.c.stats, b.c.ws)
    x, G, H, O, dO = (t.view(2, Cs, -1)[:, :n].double() for t in (b.Xp, b.G, b.H, b.O, b.dO))
    wg, w2 = W[0].double(), W[2].double()
    for name, got, ref, k in (("G", G, x @ wg.transpose(1, 2), d), ("O", O, H @ w2.transpose(1, 2), h),
                              ("dW2", dW[2], dO.transpose(1, 2) @ H, n)):
        assert rel(got, ref) <= bound(k), (name, rel(got, ref), bound(k))


def test_layer_of_short_contractions():
    """Forward and backward of a layer whose contractions have 128 to 512 values: no output further from the oracle in 64
    bits than the CUDA-core GEMMs leave it (5 % for the scatter of two errors of 7e-7)."""
    w = gw.WORKLOADS["tiny"]
    inp = gw.make_inputs(w)
    o = ob.Oracle("f64")
    x = {k: v.astype(np.float64) for k, v in inp.items() if isinstance(v, np.ndarray)}
    fw = o.forward(x["X"], x["R"], x["W1g"], x["W1u"], x["W2"], D=w.D, k=w.k, capacity=w.capacity, mode=ob.MODE_TCR)
    bw = o.backward(fw, x["X"], x["R"], x["W1g"], x["W1u"], x["W2"], x["dY"])
    dev, off = hz.upload(w, inp), []
    for impl in (etr.GEMM_AUTO, etr.GEMM_SIMT):
        cfg = hz.make_cfg(w, mode=ob.MODE_TCR, gemm_impl=impl)
        buf = etr.LayerBuffers(cfg)
        out = [torch.empty_like(t) for t in (dev.X, dev.X, dev.R, dev.W1g, dev.W1u, dev.W2)]
        etr.layer_forward(cfg, dev.X, dev.R, dev.W1g, dev.W1u, dev.W2, buf, out[0])
        etr.layer_backward(cfg, dev.X, dev.R, dev.W1g, dev.W1u, dev.W2, dev.dY, buf, *out[1:])
        assert buf.read_stats().error_word == 0
        off.append([rel(got, torch.from_numpy(np.asarray(ref)).cuda())
                    for got, ref in zip(out, (fw.Y, bw.dX, bw.dR, bw.dW1g, bw.dW1u, bw.dW2))])
    assert all(a <= 1.05 * s for a, s in zip(*off)), off


def test_repeated_passes_give_the_same_bits():
    """The same forward pass 2000 times, 32 K blocks a tile of SwiGLU and more operands than L2 holds, so that copies land late
    and out of order now and then: every bit as in the first pass (a block split before it had landed lost the lower halves of
    its operands, 1e-5 of an output, in one pass of 800)."""
    cfg, b, W = layer(52, 1000, 184, 304, (304,) * 52)
    first, differ = None, torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(2000):
        etr.expert_ffn(cfg, b.route, b.Xp, *W, b.G, b.U, b.H, b.O, b.c.stats, b.c.ws)
        got = [t.view(torch.int32) for t in (b.G, b.U, b.H, b.O)]
        first = first or [t.clone() for t in got]
        differ += torch.stack([(x != y).sum() for x, y in zip(got, first)]).sum()
    assert b.read_stats().error_word == 0
    assert int(differ) == 0
