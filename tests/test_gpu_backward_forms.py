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
    (40, 576, 256, 300, tuple((53 * i) % 301 for i in range(40))),      # more tiles than pairs, three and more per pair
    (2, 1984, 64, 260, (260, 257)),                          # the longest derivative that goes through boxes
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
