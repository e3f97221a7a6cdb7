"""The C-ABI library builds without a GPU, loads, and exports every function include/etr.h
declares; host-side argument checks work with no device present."""
import ctypes
import os
import re

from paper_2406_00023_b200 import build as etr_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    text = open(os.path.join(ROOT, "include", "etr.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(etr_[a-z0-9_]+)\s*\(", text)))


def test_library_exports_every_declared_symbol():
    lib = ctypes.CDLL(etr_build.build())
    names = declared_functions()
    assert len(names) >= 23
    for n in names:
        assert hasattr(lib, n), f"{n} declared in etr.h but not exported"


def test_binding_lists_the_same_entry_points():
    from paper_2406_00023_b200 import etr
    assert sorted(etr.EXPORTS) == declared_functions()


def test_host_side_validation_needs_no_gpu():
    from paper_2406_00023_b200 import etr
    good = etr.make_config(T=512, d=256, D=4, E=8, k=2, h=512, capacity=160, dtype=etr.F32)
    assert etr.validate(good) == etr.OK
    assert etr.c_stride(good) == 256
    assert etr.workspace_bytes(good) > 0
    assert etr.validate(etr.make_config(T=512, d=256, D=3, E=8, k=2, h=512, capacity=160, dtype=etr.F32)) == etr.ERR_SHAPE
    assert etr.validate(etr.make_config(T=512, d=256, D=4, E=8, k=9, h=512, capacity=160, dtype=etr.F32)) == etr.ERR_SHAPE
    assert etr.validate(etr.make_config(T=512, d=256, D=4, E=8, k=2, h=512, capacity=0, dtype=etr.F32)) == etr.ERR_ARG
    assert etr.validate(etr.make_config(T=512, d=256, D=4, E=8, k=2, h=512, capacity=160, dtype=5)) == etr.ERR_ARG
    assert "aligned" in etr.status_string(etr.ERR_ALIGN)
    n = ctypes.c_size_t(0)
    assert etr.lib().etr_buffers_bytes(ctypes.byref(good), 1, ctypes.byref(n)) == etr.OK and n.value > 1 << 20
    # struct layouts the binding relies on
    assert ctypes.sizeof(etr.Config) == 112 and ctypes.sizeof(etr.Stats) == 64
    # fp32 master weights under bf16 activations are taken (rounded to bf16 in the tail of the workspace, which
    # grows by three weight tensors of 2 bytes); bf16 weights under fp32 activations have no kernel
    assert etr.validate(etr.make_config(T=512, d=256, D=4, E=8, k=2, h=512, capacity=160, dtype=etr.F32,
                                        weight_dtype=etr.BF16)) == etr.ERR_UNSUPPORTED
    b16 = etr.make_config(T=512, d=256, D=4, E=8, k=2, h=512, capacity=160, dtype=etr.BF16)
    mixed = etr.make_config(T=512, d=256, D=4, E=8, k=2, h=512, capacity=160, dtype=etr.BF16, weight_dtype=etr.F32)
    assert etr.validate(mixed) == etr.OK
    assert etr.workspace_bytes(mixed) == etr.workspace_bytes(b16) + 3 * 2 * 8 * 256 * 512


def test_layout_gives_the_offsets_bind_uses():
    from paper_2406_00023_b200 import etr
    for staging, gate in ((0, etr.GATE_AFFINITY), (1, etr.GATE_SOFTMAX)):
        cfg = etr.make_config(T=512, d=256, D=4, E=8, k=2, h=512, capacity=160, dtype=etr.BF16, gate_mode=gate)
        lay = etr.layout(cfg, bool(staging))
        n = ctypes.c_size_t(0)
        assert etr.lib().etr_buffers_bytes(ctypes.byref(cfg), staging, ctypes.byref(n)) == etr.OK
        assert lay.total_bytes == n.value and lay.C_stride == 256 and lay.ws_bytes == etr.workspace_bytes(cfg)
        base = 1 << 20                                   # binding only computes addresses: no memory is touched
        b = etr.Buffers()
        assert etr.lib().etr_buffers_bind(ctypes.byref(cfg), staging, ctypes.c_void_p(base),
                                          ctypes.c_size_t(n.value), ctypes.byref(b)) == etr.OK
        for name in ("delta", "Z", "xnorm", "rnorm", "Xp", "G", "U", "H", "O", "dO", "dG", "dU", "dXp", "dgate", "ws"):
            assert getattr(b, name) == base + getattr(lay, name), name
            assert getattr(lay, name) % 256 == 0
        assert b.route.slot_token == base + lay.slot_token and b.route.tok_row == base + lay.tok_row
        assert b.stats == base + lay.stats
        if staging:
            assert b.X_dev == base + lay.X_dev and b.lse == base + lay.lse and lay.ddelta > lay.lse > 0
        else:
            assert lay.X_dev == 0 and lay.lse == 0 and not b.X_dev


def test_workspace_never_shrinks_with_the_batch():
    """Buffers made for one batch serve every shorter one: their size and that of the scratch in them never fall as T,
    E or the pooled width grows, for both gates."""
    from paper_2406_00023_b200 import etr

    def sizes(**kw):
        cfg = etr.make_config(**dict(dict(T=512, d=2048, D=8, E=32, k=2, h=64, capacity=64, dtype=etr.BF16), **kw))
        n = ctypes.c_size_t(0)
        assert etr.lib().etr_buffers_bytes(ctypes.byref(cfg), 0, ctypes.byref(n)) == etr.OK
        return etr.workspace_bytes(cfg), n.value

    for gate in (etr.GATE_AFFINITY, etr.GATE_SOFTMAX):
        for d, D, E in ((2048, 8, 32), (64, 8, 8), (1088, 8, 12), (4096, 1, 256), (512, 4, 100)):
            last = (0, 0)
            for T in sorted({*range(1, 2000), *range(2000, 70001, 31), 9471, 9472, 9473, 18944, 18945, 37888, 37889}):
                now = sizes(T=T, d=d, D=D, E=E, gate_mode=gate)
                assert now[0] >= last[0] and now[1] >= last[1], (gate, d, D, E, T)
                last = now
        for T in (3001, 9472, 60000):
            by_E = [sizes(T=T, E=E, gate_mode=gate)[0] for E in range(2, 257)]
            by_m = [sizes(T=T, d=8 * m, D=8, E=8, dtype=etr.F32, gate_mode=gate)[0] for m in range(8, 700)]
            assert by_E == sorted(by_E) and by_m == sorted(by_m)


def test_layer_calls_refuse_a_small_workspace():
    """A scratch shorter than the configuration needs is refused before anything is launched (there is no GPU here: a
    launch would fail with another status)."""
    from paper_2406_00023_b200 import etr
    big, small = (etr.make_config(T=T, d=2048, D=8, E=32, k=2, h=64, capacity=64, dtype=etr.BF16,
                                  gate_mode=etr.GATE_SOFTMAX) for T in (16384, 512))
    b, n = etr.Buffers(), ctypes.c_size_t(0)
    assert etr.lib().etr_buffers_bytes(ctypes.byref(small), 1, ctypes.byref(n)) == etr.OK
    assert etr.lib().etr_buffers_bind(ctypes.byref(small), 1, ctypes.c_void_p(1 << 20), n, ctypes.byref(b)) == etr.OK
    p, s = ctypes.c_void_p(1 << 20), ctypes.c_void_p(0)
    L, cfg, bb = etr.lib(), ctypes.byref(big), ctypes.byref(b)
    slot = etr.HostSlotC(p, p, p, p)
    assert L.etr_layer_forward(cfg, p, p, p, p, p, bb, p, s) == etr.ERR_WORKSPACE
    assert L.etr_layer_backward(cfg, p, p, p, p, p, p, bb, p, p, p, p, p, s) == etr.ERR_WORKSPACE
    assert L.etr_layer_step_host(cfg, p, p, p, p, p, p, bb, p, p, p, p, p, p, s) == etr.ERR_WORKSPACE
    assert L.etr_layer_step_host_begin(cfg, p, p, p, p, p, p, bb, ctypes.byref(slot), ctypes.c_int32(0), p, p, p, p,
                                       p, p, s) == etr.ERR_WORKSPACE
