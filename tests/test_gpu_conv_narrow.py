"""The mma.sync convolution on narrow images (tiles of pixels in the batch's order) against
the row kernel on the same images with zero columns beside them, which takes the same sums
in the same order: bit for bit; and the transposed convolution and its data gradient on
CUDA cores with channels and pixels that fill no tile.  Needs a GB300."""
import numpy as np
import pytest

from test_gpu_conv import bf16_round, lib, run_conv, run_upback, run_upconv  # noqa: F401

pytestmark = pytest.mark.gpu


# one pixel; a tile's remainder and a tile; rows of several images in one tile; the widest
@pytest.mark.parametrize("B, H, W, cin, cout", [(1, 1, 1, 64, 32), (1, 11, 3, 64, 64), (1, 8, 4, 256, 128),
                                                (3, 5, 7, 128, 256), (2, 33, 32, 64, 128)])
def test_narrow_convolution_is_the_row_kernels(lib, B, H, W, cin, cout):  # noqa: F811
    rng = np.random.default_rng(B * H * W + cin + cout)
    x = bf16_round(rng.standard_normal((B, H, W, cin + 8)))
    Wt = bf16_round(rng.standard_normal((cout, 3, 3, cin)) * 0.05)
    bias = rng.standard_normal(cout).astype(np.float32)
    wide = np.zeros((B, H, 130, cin + 8))
    wide[:, :, :W] = x
    y, st = run_conv(lib, 1, x, 8, cin, Wt, bias, True, cout + 8, 8)
    assert st == lib.PIC_OK
    ref, st = run_conv(lib, 1, wide, 8, cin, Wt, bias, True, cout + 8, 8)
    assert st == lib.PIC_OK
    assert np.array_equal(y, ref[:, :, :W])      # the channels before the offset too: untouched


@pytest.mark.parametrize("B, h, w, cin, cout", [(1, 1, 1, 1, 1), (2, 3, 5, 33, 5), (1, 4, 4, 64, 32), (3, 1, 7, 70, 65)])
def test_transposed_convolution_on_cuda_cores(lib, B, h, w, cin, cout):  # noqa: F811
    # FP32 sums of K products and one rounding to BF16
    rng = np.random.default_rng(B + h + w + cin + cout)
    x = bf16_round(rng.standard_normal((B, h, w, cin)))
    Wup = (rng.standard_normal((2, 2, cin, cout)) * 0.1).astype(np.float32)
    bias = rng.standard_normal(cout).astype(np.float32)
    W64 = Wup.astype(np.float64)
    y, st = run_upconv(lib, 1, x, Wup, bias, cout + 3, 3)
    assert st == lib.PIC_OK
    ref = (np.einsum("bhwi,acio->bhawco", x, W64) + bias).reshape(B, 2 * h, 2 * w, cout)
    mag = (np.einsum("bhwi,acio->bhawco", abs(x), abs(W64)) + abs(bias)).reshape(ref.shape)
    assert np.all(abs(y[..., 3:] - ref) <= (cin + 1) * 2.0 ** -24 * mag + 2.0 ** -8 * abs(ref))
    g = bf16_round(rng.standard_normal((B, 2 * h, 2 * w, cout + 3)))
    gi, st = run_upback(lib, 1, g, 3, cout, Wup, cin)
    assert st == lib.PIC_OK
    g6 = g[..., 3:].reshape(B, h, 2, w, 2, cout)
    ref = np.einsum("bhawco,acio->bhwi", g6, W64)
    mag = np.einsum("bhawco,acio->bhwi", abs(g6), abs(W64))
    assert np.all(abs(gi - ref) <= 4 * cout * 2.0 ** -24 * mag + 2.0 ** -8 * abs(ref))
