"""The weight gradient's row kernel where its segments, boxes and accumulators
begin and end, against the FP64 oracle with the bounds of test_gpu_conv.py.
Needs a GB300."""
import numpy as np
import pytest

from oracle import unet as ounet
from test_gpu_conv import bf16_round, run_wgrad

pytestmark = pytest.mark.gpu

CASES = [
    # B, H, W, cin, cout, in_cs, in_off
    (1, 1, 1, 32, 32, 32, 0),            # one K block: one accumulator, one row, boxes mostly off the image
    (1, 2, 65, 64, 64, 64, 0),           # a column of one pixel
    (3, 11, 64, 32, 32, 64, 32),         # columns of odd length, an input slice
    (2, 1300, 64, 64, 64, 64, 0),        # several segments a CTA, some across images
    (1, 3700, 70, 32, 32, 32, 0),        # the same, of 14 rows and two accumulators
    (1, 2500, 64, 64, 32, 64, 0),
    (1, 1000, 130, 32, 64, 32, 0),
    (1, 2000, 64, 16, 32, 16, 0),
    (5, 7, 16, 256, 256, 256, 0),        # 16 blocks: two waves
    (1, 9, 20, 320, 192, 320, 0),        # 15 blocks
]


@pytest.mark.parametrize("case", CASES)
def test_weight_gradient_rows(case):
    import paper_1610_03918_gb300 as pg
    B, H, W, cin, cout, in_cs, in_off = case
    rng = np.random.default_rng(cin * 7 + cout * 3 + W + H)
    x_full = bf16_round(rng.standard_normal((B, H, W, in_cs)))
    dpre = bf16_round(rng.standard_normal((B, H, W, cout)))
    got, st = run_wgrad(pg, 0, dpre, x_full, in_off, cin)
    assert st == pg.PIC_OK, pg.pic_strerror(st)
    _, ref, _ = ounet.conv3x3_backward(x_full[..., in_off:in_off + cin], np.zeros((cout, 3, 3, cin)), dpre)
    # exact products; sums of B H W of them in FP32 (truncated by the tensor core)
    assert np.linalg.norm(got - ref) <= 1e-4 * np.linalg.norm(ref)
    assert np.all(np.abs(got - ref) <= 1e-3 * np.abs(ref).max())
