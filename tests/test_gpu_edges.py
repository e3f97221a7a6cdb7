"""Edge cases of the CUDA path against the oracle: experts that receive no token, Top-1
routing (the paper's efficiency runs), k = E, capacity 1, a handful of tokens, group
sizes that take the generic pooling path, and tokens with more rows than the gather kernels stage."""
import numpy as np
import pytest
import torch

from gen import workloads as gw
from oracle import binding as ob
from tests import harness as hz

pytestmark = pytest.mark.gpu
etr = hz.etr
W = gw.WORKLOADS


def layer_vs_oracle(w, inp, mode, impl=etr.GEMM_AUTO):
    o = ob.Oracle("f32")
    fw = o.forward(inp["X"], inp["R"], inp["W1g"], inp["W1u"], inp["W2"], D=w.D, k=w.k,
                   capacity=w.capacity, mode=mode)
    bw = o.backward(fw, inp["X"], inp["R"], inp["W1g"], inp["W1u"], inp["W2"], inp["dY"])
    cfg = hz.make_cfg(w, mode=mode, gemm_impl=impl)
    dev = hz.upload(w, inp)
    buf = etr.LayerBuffers(cfg)
    out = dict(Y=torch.empty_like(dev.X), dX=torch.empty_like(dev.X), dR=torch.empty_like(dev.R),
               dW1g=torch.full_like(dev.W1g, float("nan")), dW1u=torch.full_like(dev.W1u, float("nan")),
               dW2=torch.full_like(dev.W2, float("nan")))
    etr.layer_forward(cfg, dev.X, dev.R, dev.W1g, dev.W1u, dev.W2, buf, out["Y"])
    etr.layer_backward(cfg, dev.X, dev.R, dev.W1g, dev.W1u, dev.W2, dev.dY, buf, out["dX"], out["dR"],
                       out["dW1g"], out["dW1u"], out["dW2"])
    torch.cuda.synchronize()
    assert buf.read_stats().error_word == 0
    got = hz.route_from_buffers(buf, cfg)
    hz.check_route_structure(hz.to_np(buf.delta), got, mode)
    identical = hz.assert_routes_match(fw.delta, fw.route, got, mode)
    assert identical, "these cases are built with clear margins"
    tol = 2e-2 if w.dtype == "bf16" else 1e-4
    for nm, ref, chain in (("Y", fw.Y, 4), ("dX", bw.dX, 6), ("dR", bw.dR, 4), ("dW1g", bw.dW1g, 6),
                           ("dW1u", bw.dW1u, 6), ("dW2", bw.dW2, 4)):
        hz.assert_close_rms(hz.to_np(out[nm]), ref, tol, nm, chain=chain)
    return fw, got, out


TC_FORMS = [etr.GEMM_TCGEN05, etr.GEMM_TCGEN05_2CTA, etr.GEMM_TCGEN05_2CTA_WIDE]


@pytest.mark.parametrize("dtype,impl", [("f32", etr.GEMM_AUTO), ("bf16", etr.GEMM_AUTO), ("bf16", etr.GEMM_SIMT)]
                         + [("bf16", f) for f in TC_FORMS])
def test_experts_without_tokens_get_zero_gradients(dtype, impl):
    """Token choice with every token pushed away from experts 2 and 5: their buffers stay
    empty, their weight gradients must be exactly zero, everything else must match."""
    w = gw.scaled(W["small"], T=384, d=256, D=8, E=8, h=128, dtype=dtype)
    inp = gw.make_inputs(w)
    lean = np.repeat(inp["R"], w.D, axis=1)              # expert directions in R^d
    X = inp["X"] - 0.5 * (lean[2] + lean[5])[None, :] * np.sqrt(w.d / w.D)
    inp["X"] = gw.round_to_bf16(X) if dtype == "bf16" else X.astype(np.float32)
    fw, got, out = layer_vs_oracle(w, inp, ob.MODE_TCR, impl)
    assert got.counts[2] == 0 and got.counts[5] == 0 and got.counts.sum() > 0
    for nm in ("dW1g", "dW1u", "dW2"):
        g = out[nm]
        assert bool((g[2] == 0).all()) and bool((g[5] == 0).all()), nm
    assert bool((out["dR"][2] == 0).all())


@pytest.mark.parametrize("impl", [etr.GEMM_AUTO] + TC_FORMS)
@pytest.mark.parametrize("k", [1, 8])
def test_top1_and_top_all(k, impl):
    """h = 192 and d = 256 leave ragged column tiles in every tile form."""
    w = gw.scaled(W["small"], T=300, d=256, D=8, E=8, h=192, k=k, cf=0.8)
    layer_vs_oracle(w, gw.make_inputs(w), ob.MODE_TCR, impl)


@pytest.mark.parametrize("impl", [etr.GEMM_AUTO] + TC_FORMS)
@pytest.mark.parametrize("mode", [ob.MODE_TCR, ob.MODE_ECR])
def test_capacity_one_and_few_tokens(mode, impl):
    w = gw.scaled(W["small"], T=5, d=128, D=8, E=4, h=64, cf=0.2)
    assert w.capacity == 1
    layer_vs_oracle(w, gw.make_inputs(w), mode, impl)


@pytest.mark.parametrize("impl", TC_FORMS)
def test_wide_columns_with_a_ragged_second_half(impl):
    """d = 640 and h = 320: the 512-column tiles of the wide form end in a partial second half
    (640 = 512 + 128) or have none at all (320), with 700 tokens per expert at most (ragged rows)."""
    w = gw.scaled(W["small"], T=1400, d=640, D=8, E=4, h=320, cf=1.0)
    layer_vs_oracle(w, gw.make_inputs(w), ob.MODE_ECR, impl)


@pytest.mark.parametrize("D,dtype", [(1, "f32"), (2, "bf16"), (4, "bf16"), (32, "bf16"), (24, "f32")])
def test_group_sizes(D, dtype):
    """D = 1 (plain cosine routing), sub-vector groups, wide groups and a group size that is
    neither a divisor nor a multiple of 8."""
    d = 768 if D == 24 else 512
    w = gw.scaled(W["small"], T=200, d=d, D=D, E=8, h=64, dtype=dtype)
    layer_vs_oracle(w, gw.make_inputs(w), ob.MODE_TCR)


@pytest.mark.parametrize("T,E,d,D,h,dtype", [
    (40, 128, 1024, 8, 64, "bf16"), (40, 128, 1024, 8, 64, "f32"),
    (2400, 72, 584, 8, 8, "f32"),                            # 576 entries a block in both kernels
    (4747, 40, 320, 8, 64, "bf16"), (4747, 40, 328, 8, 8, "f32"), (4747, 40, 168, 4, 8, "f32"),      # R gathered beside the rows
    (4747, 40, 200, 5, 8, "f32"),                            # any other group size: through shared memory
])
def test_tokens_kept_by_every_expert_overflow_the_staged_row_lists(T, E, d, D, h, dtype):
    """Expert choice with C = T: every token has a row of every expert.  The combine kernel takes up to 8 tokens a block and the
    fused dX kernel up to 16, as many as leave every SM two blocks, and each stages 512 row entries in shared memory: the
    entries beyond are read in place.  2400 tokens: 8 a block in both.  4747: 16 in dX, the last block 11.  40 tokens are one
    and two a block, whose 128 and 256 entries fit.  (The router's part of dX, which the entries beyond enter in two ways, is
    over half of dX here.)"""
    w = gw.scaled(W["small"], T=T, d=d, D=D, E=E, h=h, cf=E / 2, dtype=dtype)
    assert w.capacity == w.T
    if T > 40:
        two_a_sm = 2 * torch.cuda.get_device_properties(0).multi_processor_count
        assert (T // 8 >= two_a_sm and 8 * E > 512) or (T // 16 >= two_a_sm and 16 * E > 512)
    fw, got, out = layer_vs_oracle(w, gw.make_inputs(w), ob.MODE_ECR)
    assert np.all(np.diff(got.tok_ptr) == w.E)


@pytest.mark.parametrize("d,D,dtype,T,C", [
    (2048, 16, "bf16", 215, 54), (2048, 4, "bf16", 215, 54), (2048, 8, "f32", 215, 54), (4096, 32, "bf16", 215, 54),
    (8192, 64, "bf16", 215, 54),
    # capacities whose cuts leave at least 1e-5 between the last affinity kept and the first one not
    (512, 8, "bf16", 4747, 1042), (512, 4, "f32", 4747, 1114), (512, 2, "bf16", 4747, 1177),
])
def test_fused_dx_at_wide_hidden_sizes(d, D, dtype, T, C):
    """Hidden sizes of 2048, 4096 and 8192 in the fused dX kernel (whole 4 to 16 KiB rows per token and row of dXp),
    power-of-two and generic group sizes, and expert choice with C of about T / 4, which gives tokens anything from no row
    (zeros, X not read) to the rows of most of the 16 experts.  215 tokens are two a block, the last one alone; 4747 are 16 a
    block (the last 11), whose list of row entries crosses many token boundaries."""
    w = gw.scaled(W["small"], T=T, d=d, D=D, E=16, h=64, cf=(C - 0.5) * 8 / T, dtype=dtype)
    assert w.capacity == C
    fw, got, out = layer_vs_oracle(w, gw.make_inputs(w), ob.MODE_ECR)
    n = np.diff(got.tok_ptr)
    assert n.min() == 0 and n.max() >= 6 and n.sum() > 3 * w.T


def _affinity_on_device(w, inp, rows=None):
    cfg = hz.make_cfg(w if rows is None else gw.scaled(w, T=rows.stop - rows.start))
    X = hz.to_dev(inp["X"] if rows is None else inp["X"][rows], w)
    R = torch.from_numpy(inp["R"]).cuda()
    T, m = X.shape[0], w.d // w.D
    delta = torch.empty(T, w.E, dtype=torch.float32, device="cuda")
    Z = torch.empty(T, m, dtype=torch.float32, device="cuda")
    xnorm = torch.empty(T, dtype=torch.float32, device="cuda")
    rnorm = torch.empty(w.E, dtype=torch.float32, device="cuda")
    stats = torch.zeros(16, dtype=torch.int32, device="cuda")
    etr.affinity(cfg, X, R, delta, Z, xnorm, rnorm, stats)
    torch.cuda.synchronize()
    assert int(stats[6].item()) == 0            # error_word
    return delta, rnorm, stats


@pytest.mark.parametrize("T,d,D,E,dtype", [(1000, 256, 8, 7, "bf16"), (130, 512, 4, 64, "f32"), (4097, 2048, 8, 33, "bf16"),
                                            (127, 64, 2, 1, "bf16"), (20000, 1024, 4, 12, "bf16")])
def test_affinity_scores_on_the_tensor_cores(T, d, D, E, dtype):
    """Shapes the tensor-core score kernel takes (E <= 64, 32 | d/D): expert counts that are not a multiple of 4
    (scalar stores), a single expert, one K block, a ragged last tile of tokens, more tiles than SMs.  Affinities
    within the usual 1e-5, the batch maximum equal to the largest affinity stored, and a token's affinities the
    same bits whether it is scored in the whole batch or in a slice of it."""
    w = gw.scaled(W["small"], T=T, d=d, D=D, E=E, k=1, h=64, dtype=dtype)
    assert E <= 64 and (d // D) % 32 == 0
    inp = gw.make_inputs(w, weights=False)
    delta_ref, _, rnorm_ref, _ = ob.Oracle("f32").affinity(inp["X"], inp["R"], w.D)
    delta, rnorm, stats = _affinity_on_device(w, inp)
    got = hz.to_np(delta)
    hz.assert_affinity_close(got, delta_ref)
    assert np.allclose(hz.to_np(rnorm), rnorm_ref, rtol=1e-6, atol=0)
    u = int(np.float32(got.max()).view(np.uint32))
    key = (~u & 0xffffffff) if (u & 0x80000000) else (u | 0x80000000)
    assert int(stats[5].item()) & 0xffffffff == key
    rows = slice(T // 3, T // 3 + min(300, T - T // 3))
    part, _, _ = _affinity_on_device(w, inp, rows)
    assert torch.equal(part, delta[rows])


@pytest.mark.parametrize("E,dtype,d", [(16, "bf16", 640), (32, "f32", 640), (64, "bf16", 640), (64, "bf16", 512)])
def test_affinity_with_a_score_tile_for_every_sm(E, dtype, d):
    """38100 tokens: at least one 256-token tile per SM and a ragged last tile.  With d/D = 80 (16 divides it, 32
    does not) the fp32 score kernel takes its register-tiled form (2, 4 or 8 experts per lane for E <= 16, 32,
    64); with d/D = 64 the tensor-core kernel takes the same batch."""
    w = gw.scaled(W["small"], T=38100, d=d, D=8, E=E, h=64, dtype=dtype)
    inp = gw.make_inputs(w, weights=False)
    delta_ref, *_ = ob.Oracle("f32").affinity(inp["X"], inp["R"], w.D)
    cfg = hz.make_cfg(w)
    X = hz.to_dev(inp["X"], w)
    R = torch.from_numpy(inp["R"]).cuda()
    T, m = w.T, w.d // w.D
    delta = torch.empty(T, E, dtype=torch.float32, device="cuda")
    Z = torch.empty(T, m, dtype=torch.float32, device="cuda")
    xnorm = torch.empty(T, dtype=torch.float32, device="cuda")
    rnorm = torch.empty(E, dtype=torch.float32, device="cuda")
    stats = torch.zeros(16, dtype=torch.int32, device="cuda")
    etr.affinity(cfg, X, R, delta, Z, xnorm, rnorm, stats)
    torch.cuda.synchronize()
    got = hz.to_np(delta)
    hz.assert_affinity_close(got, delta_ref)
    u = int(np.float32(got.max()).view(np.uint32))
    key = (~u & 0xffffffff) if (u & 0x80000000) else (u | 0x80000000)
    assert int(stats[5].item()) & 0xffffffff == key


def test_sweep_modes_follow_the_step():
    """ETR_MODE_AUTO picks token choice before switch_step and expert choice from it on."""
    for step, want in ((999, etr.MODE_TCR), (1000, etr.MODE_ECR)):
        w = gw.scaled(W["sweep"], T=256, d=256, D=16, E=8, h=64, n_clusters=8, step=step)
        inp = gw.make_inputs(w)
        cfg = etr.make_config(T=w.T, d=w.d, D=w.D, E=w.E, k=w.k, h=w.h, capacity=w.capacity,
                              dtype=etr.BF16, mode=etr.MODE_AUTO, step=step, switch_step=w.switch_step,
                              adaptive=True)
        dev = hz.upload(w, inp)
        buf = etr.LayerBuffers(cfg)
        Y = torch.empty_like(dev.X)
        etr.layer_forward(cfg, dev.X, dev.R, dev.W1g, dev.W1u, dev.W2, buf, Y)
        st = buf.read_stats()
        assert st.mode == want and 1 <= st.C <= w.capacity
        o = ob.Oracle("f32")
        delta, *_ = o.affinity(inp["X"], inp["R"], w.D)
        assert st.C == ob.capacity_bound(w.d, w.E, w.capacity, 1, True, st.delta_max)
        if want == etr.MODE_ECR:
            assert np.all(hz.to_np(buf.counts) == min(st.C, w.T))


@pytest.mark.parametrize("d,D", [(2560, 4), (2432, 4), (3072, 4), (2368, 4), (4096, 4), (1216, 1)])
def test_pooled_widths_at_the_shared_memory_limit_of_the_fused_dx_kernel(d, D):
    """608 to 768 (and 1216 to 1536) pooled columns: cz of 16 (8) tokens together with the row lists is more shared
    memory than a launch gets without opting in."""
    w = gw.scaled(W["small"], T=70, d=d, D=D, E=4, h=64)
    layer_vs_oracle(w, gw.make_inputs(w), ob.MODE_TCR)


@pytest.mark.parametrize("d,D,T", [(264, 8, 300), (24, 1, 150), (1312, 1, 140), (520, 4, 700)])
def test_router_gradient_sums_at_the_edges_of_their_groups(d, D, T):
    """33, 24, 1312 and 130 pooled columns: rows of Z that are no multiple of 16 bytes, shorter than a warp, longer than
    a block, and of a width that leaves threads over; chunks of 128 slots that end inside (fp32, 1e-4)."""
    w = gw.scaled(W["small"], T=T, d=d, D=D, E=4, h=64, dtype="f32")
    layer_vs_oracle(w, gw.make_inputs(w), ob.MODE_TCR)


@pytest.mark.parametrize("gate", [etr.GATE_AFFINITY, etr.GATE_SOFTMAX])
def test_buffers_of_a_longer_batch_serve_a_shorter_one(gate):
    """A step of 9000 tokens on buffers made for 16384 gives the bits of buffers made for 9000 (the dense router
    gradient cuts the shorter batch into more chunks than the longer one)."""
    T, d, D, E, h = 9000, 2048, 8, 32, 64
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    X, dY = rnd(T, d).bfloat16(), rnd(T, d).bfloat16()
    R = rnd(E, d // D)
    W1g, W1u, W2 = ((rnd(*s) / d ** 0.5).bfloat16() for s in ((E, h, d), (E, h, d), (E, d, h)))
    short, longer = (etr.make_config(T=n, d=d, D=D, E=E, k=2, h=h, capacity=700, dtype=etr.BF16, mode=etr.MODE_TCR,
                                     gate_mode=gate) for n in (T, 16384))
    outs = []
    for made_for in (short, longer):
        buf = etr.LayerBuffers(made_for)
        out = [torch.empty_like(t) for t in (X, X, R, W1g, W1u, W2)]
        etr.layer_forward(short, X, R, W1g, W1u, W2, buf, out[0])
        etr.layer_backward(short, X, R, W1g, W1u, W2, dY, buf, *out[1:])
        assert buf.read_stats().error_word == 0
        outs.append(out)
    assert all(torch.equal(a, b) for a, b in zip(*outs))


def test_layer_backward_takes_pooled_tokens_at_any_float_address():
    """The backward layer call reads Z where the caller has put it, here one float behind a 16-byte boundary: the sums
    of dR are taken in another order (fp32 sums of at most 160 products: 1e-6), everything else has the same bits."""
    w = gw.scaled(W["small"], T=512, d=256, D=4, E=8, h=64, dtype="f32")
    inp = gw.make_inputs(w)
    cfg, dev = hz.make_cfg(w, mode=ob.MODE_TCR), hz.upload(w, inp)
    buf = etr.LayerBuffers(cfg)
    Y = torch.empty_like(dev.X)
    etr.layer_forward(cfg, dev.X, dev.R, dev.W1g, dev.W1u, dev.W2, buf, Y)
    outs = []
    shifted = torch.empty(buf.Z.numel() + 1, device="cuda")
    shifted[1:].copy_(buf.Z.flatten())
    for Z in (buf.c.Z, shifted.data_ptr() + 4):
        buf.c.Z = Z
        outs.append([torch.empty_like(t) for t in (dev.X, dev.R, dev.W1g, dev.W1u, dev.W2)])
        etr.layer_backward(cfg, dev.X, dev.R, dev.W1g, dev.W1u, dev.W2, dev.dY, buf, *outs[-1])
    torch.cuda.synchronize()
    for i, (a, b) in enumerate(zip(*outs)):
        assert float((a - b).norm()) <= 1e-6 * float(a.norm()) if i == 1 else torch.equal(a, b)
