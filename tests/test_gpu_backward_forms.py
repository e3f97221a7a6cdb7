"""Weight gradients (one launch for the three, outputs stored through boxes) and the SwiGLU derivative (G and U fetched, dG and
dU stored through boxes), as AUTO runs them, bit for bit against the single-CTA form, which runs each gradient by itself and
stores from the warps: the same products in the same order, so no tolerance.  Every buffer starts as NaN: what a launch leaves
out, or writes outside its rows, shows."""
import pytest
import torch

from paper_2406_00023_b200 import etr
from test_gpu_swapped_gemm import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grad_fp32", [False, True])
@pytest.mark.parametrize("E,d,h,cap,counts", [
    (3, 64, 64, 16, (16, 0, 1)),                             # K blocks of 16 rows; one block of 64 columns either way
    (2, 192, 320, 17, (17, 16)),                             # of 32; last column tiles of 64 and 192 columns
    (2, 320, 128, 33, (33, 32)),                             # of 64, the last one with one row
    (4, 256, 640, 200, (200, 0, 65, 129)),                   # whole tiles and a last one of 128 columns
    (40, 576, 256, 300, tuple((53 * i) % 301 for i in range(40))),      # 360 tiles of gradients, four and five a pair
    (2, 1984, 64, 260, (260, 257)),                          # the longest derivative that goes through boxes (4 tiles)
    (2, 2048, 64, 260, (260, 257)),                          # the shortest that does not
])
def test_against_the_single_cta_form(E, d, h, cap, counts, grad_fp32):
    a, _, _, dWa = run(E, d, h, cap, counts, etr.GEMM_AUTO, grad_fp32)
    b, _, _, dWb = run(E, d, h, cap, counts, etr.GEMM_TCGEN05, grad_fp32)
    for x, y in zip(dWa, dWb):
        assert torch.equal(x, y) and bool(torch.isfinite(x).all())
    for name in ("G", "U", "H", "dG", "dU"):
        x, y = getattr(a, name).view(torch.int16), getattr(b, name).view(torch.int16)
        assert torch.equal(x, y), name


@pytest.mark.parametrize("E,d,h,cap,counts", [
    (40, 320, 320, 600, (600,) * 40),                        # 240 tiles, half of them with 64 columns
    (64, 256, 576, 300, tuple(257 + (11 * i) % 44 for i in range(64))),  # 384, a third of them with 64; second row tiles of 1 to 44 rows
    (128, 128, 64, 520, tuple((67 * i) % 521 for i in range(128))),      # 192, every one with 64; an expert without rows
    (40, 320, 448, 600, (600,) * 40),                        # 240, half of them with 192
    (40, 320, 384, 600, (600,) * 40),                        # 240, half of them with 128
    (64, 256, 512, 300, (300, 0, 1, 257) * 16),              # whole columns, 0 to 2 row tiles an expert
])
def test_derivative_tiles_that_use_an_accumulator_again(E, d, h, cap, counts):
    """The SwiGLU derivative on pairs with three tiles and more, whose two accumulators are used again, behind last
    column tiles of every width: each of the 16 epilogue warps gives each accumulator back once per tile, also where it has no
    column or no row of it.  Waits are cut to some 50 ms: a return that is missed ends in the error word that `run` checks."""
    limit = 100_000_000
    tiles = sum((n + 255) // 256 for n in counts) * ((h + 255) // 256)
    assert tiles > 2 * 74 and cap > 192 and d < 2048         # more than two tiles a pair; rules of the forms
    a, _, _, dWa = run(E, d, h, cap, counts, etr.GEMM_AUTO, wait_limit_cycles=limit)
    b, _, _, dWb = run(E, d, h, cap, counts, etr.GEMM_TCGEN05, wait_limit_cycles=limit)
    for name in ("dG", "dU", "dXp"):
        assert torch.equal(getattr(a, name).view(torch.int16), getattr(b, name).view(torch.int16)), name
    assert all(torch.equal(x, y) for x, y in zip(dWa, dWb))


def test_fp32_master_step_with_a_last_column_tile_of_64():
    """A whole step of a layer with fp32 weights at h = 1344 = 5 * 256 + 64, four tiles of the derivative per pair."""
    T, d, E, h = 6000, 256, 24, 1344
    g = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    X, dY, R = rnd(T, d).bfloat16(), rnd(T, d).bfloat16(), rnd(E, d // 8)
    W = [rnd(*s) / s[2] ** 0.5 for s in ((E, h, d), (E, h, d), (E, d, h))]
    outs = []
    for impl in (etr.GEMM_AUTO, etr.GEMM_TCGEN05):
        cfg = etr.make_config(T=T, d=d, D=8, E=E, k=2, h=h, capacity=625, dtype=etr.BF16, mode=etr.MODE_ECR, gemm_impl=impl,
                              weight_dtype=etr.F32, grad_fp32=True, wait_limit_cycles=100_000_000)
        buf = etr.LayerBuffers(cfg)
        out = [torch.full_like(t, float("nan")) for t in (X, X, R, *W)]
        etr.layer_forward(cfg, X, R, *W, buf, out[0])
        etr.layer_backward(cfg, X, R, *W, dY, buf, *out[1:])
        assert buf.read_stats().error_word == 0
        outs.append(out)
    assert all(torch.equal(x, y) and bool(torch.isfinite(x).all()) for x, y in zip(*outs))
