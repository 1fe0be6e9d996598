"""The transposed convolution's bias gradient for every channel count its tensor-core
route takes, also one whose groups of eight do not divide a CTA (192): against an FP64
sum.  Needs a GB300."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cout", [32, 64, 128, 192, 256])
@pytest.mark.parametrize("B, H, W", [(1, 1, 1), (2, 9, 24), (3, 37, 41)])
def test_bias_gradient(B, H, W, cout):
    import torch
    import paper_1610_03918_gb300 as pg
    P, I = ctypes.c_void_p, ctypes.c_int32
    f = pg.load_library().pic_upconv_wgrad_bf16
    f.argtypes, f.restype = [I, I, I, I, P, I, P, I, I, I, P, P, P], ctypes.c_int
    g = torch.Generator(device="cuda").manual_seed(cout + H)
    x = torch.randn((B, H, W, 64), generator=g, device="cuda").bfloat16()
    dy = torch.randn((B, 2 * H, 2 * W, cout), generator=g, device="cuda").bfloat16()
    dw, db = torch.zeros(4 * 64 * cout, device="cuda"), torch.zeros(cout, device="cuda")
    assert f(0, B, H, W, x.data_ptr(), 64, dy.data_ptr(), cout, 0, cout, dw.data_ptr(), db.data_ptr(),
             torch.cuda.current_stream().cuda_stream) == pg.PIC_OK
    # FP32 sums of at most 4 B H W terms: the error of n additions in any order is below
    # n 2^-24 of the sum of the magnitudes
    ref, mag, n = dy.double().sum((0, 1, 2)), dy.double().abs().sum((0, 1, 2)), 4 * B * H * W
    assert bool(((db.double() - ref).abs() <= n * 2.0 ** -24 * mag).all())
