"""The persistent row kernel of the 3x3 convolution (images at least 128
pixels wide) at the sizes where its runs, ring and stores can go wrong, against
the FP64 oracle with the single-layer bounds of test_gpu_conv.py.  Needs a
GB300."""
import numpy as np
import pytest

from oracle import unet as ounet
from test_gpu_conv import bf16_round, run_conv

pytestmark = pytest.mark.gpu

CASES = [
    # B, H, W, cin, cout, in_cs, in_off, out_cs, out_off, relu
    (1, 1, 128, 32, 32, 32, 0, 32, 0, True),        # one output row: a run of one
    (3, 29, 300, 32, 32, 64, 32, 96, 32, True),     # ragged column block, channel slices, runs across images
    (1, 700, 130, 32, 32, 32, 0, 32, 0, False),     # more rows than CTAs; a column block of two pixels
    (2, 4, 256, 32, 64, 32, 0, 72, 8, True),        # 16-byte stores (stride no multiple of 16)
    (1, 333, 140, 64, 32, 64, 0, 32, 0, True),
    (2, 37, 129, 64, 64, 128, 64, 64, 0, True),
    (1, 151, 256, 128, 64, 128, 0, 64, 0, True),    # two channel blocks, a unit per vertical tap
    (1, 160, 128, 128, 128, 128, 0, 256, 128, True),    # tap order, two column halves
    (1, 9, 130, 128, 128, 128, 0, 128, 0, False),   # few tiles
    (1, 200, 128, 64, 128, 64, 0, 128, 0, True),
    (1, 5, 200, 128, 256, 128, 0, 256, 0, True),    # four column blocks
    (1, 6, 128, 256, 128, 256, 0, 128, 0, True),    # four channel blocks, few tiles
    (2, 90, 160, 256, 128, 256, 0, 256, 0, False),  # and in tap order
    (1, 3, 128, 64, 64, 64, 0, 64, 0, True),        # runs of a row or two
]


@pytest.mark.parametrize("case", CASES)
def test_row_kernel_matches_oracle(case):
    import paper_1610_03918_gb300 as pg
    B, H, W, cin, cout, in_cs, in_off, out_cs, out_off, relu = case
    rng = np.random.default_rng(cin * 1000 + cout + H + W)
    x_full = bf16_round(rng.standard_normal((B, H, W, in_cs)))
    Wt = bf16_round(rng.standard_normal((cout, 3, 3, cin)) * np.sqrt(2.0 / (9 * cin)))
    bias = rng.standard_normal(cout) * 0.1
    out, st = run_conv(pg, 0, x_full, in_off, cin, Wt, bias, relu, out_cs, out_off)
    assert st == pg.PIC_OK, pg.pic_strerror(st)
    ref = ounet.conv3x3(x_full[..., in_off:in_off + cin], Wt, bias)
    if relu:
        ref = np.maximum(ref, 0.0)
    got = out[..., out_off:out_off + cout]
    rel = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert rel <= 4e-3, rel
    assert np.all(np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-3 * np.abs(ref).max())
    rest = np.delete(out, np.s_[out_off:out_off + cout], axis=3)
    assert np.all(rest == 7.0)   # channels outside the output slice are untouched


@pytest.mark.parametrize("W, cin, cout", [(40, 64, 64), (9, 32, 256), (200, 16, 32)])
def test_store_width_changes_no_result(W, cin, cout):
    # the tile kernel stores 16 channels in one piece where they are 32-byte
    # aligned (offset 0) and in two where not (offset 8): the same bits
    import paper_1610_03918_gb300 as pg
    rng = np.random.default_rng(W + cin)
    x = bf16_round(rng.standard_normal((2, 13, W, cin)))
    Wt = bf16_round(rng.standard_normal((cout, 3, 3, cin)) * 0.1)
    bias = rng.standard_normal(cout) * 0.1
    wide, st = run_conv(pg, 0, x, 0, cin, Wt, bias, True, cout, 0)
    assert st == pg.PIC_OK
    for cs, off in ((cout + 8, 8), (cout + 8, 0), (cout + 16, 8)):
        out, st = run_conv(pg, 0, x, 0, cin, Wt, bias, True, cs, off)
        assert st == pg.PIC_OK
        assert np.array_equal(out[..., off:off + cout], wide)
        assert np.all(np.delete(out, np.s_[off:off + cout], axis=3) == 7.0)


@pytest.mark.parametrize("H, W, cin, cout", [
    (5, 24, 64, 32), (3, 130, 128, 64), (4, 64, 256, 128),
    (40, 300, 64, 32),      # several tiles a CTA, a ragged column block
    (97, 128, 128, 64),     # 256 columns at once
    (1, 8, 32, 16),         # a part of one tile; 64 columns, K = 32
    (33, 9, 96, 32),        # three units, tiles of 8 x 16 pixels
    (70, 90, 256, 128),     # 512 columns
])
def test_upconv_store_width_changes_no_result(H, W, cin, cout):
    import ctypes
    import torch
    import paper_1610_03918_gb300 as pg
    f = pg.load_library().pic_upconv_bf16
    f.argtypes = [ctypes.c_int32] * 4 + [ctypes.c_void_p, ctypes.c_int32] + [ctypes.c_void_p] * 3 \
        + [ctypes.c_int32] * 3 + [ctypes.c_void_p]
    g = torch.Generator(device="cuda").manual_seed(H + W)
    x = torch.randn((2, H, W, cin), generator=g, device="cuda").bfloat16()
    w = torch.randn((2, 2, cin, cout), generator=g, device="cuda")
    b = torch.randn((cout,), generator=g, device="cuda")
    outs = []
    for cs, off in ((cout, 0), (2 * cout, cout), (cout + 8, 8)):
        out = torch.full((2, 2 * H, 2 * W, cs), 7.0, device="cuda").bfloat16()
        assert f(0, 2, H, W, x.data_ptr(), cin, w.data_ptr(), b.data_ptr(), out.data_ptr(), cs, off, cout,
                 torch.cuda.current_stream().cuda_stream) == pg.PIC_OK
        outs.append(out[..., off:off + cout].clone())
        out[..., off:off + cout] = 7.0
        assert bool((out == 7.0).all())
    ref = torch.einsum("bhwi,acio->bhawco", x.double(), w.bfloat16().double()).reshape(2, 2 * H, 2 * W, cout) + b
    # FP32 sums of cin products and one rounding to BF16
    assert float((outs[0].double() - ref).norm() / ref.norm()) <= 4e-3
    assert all(torch.equal(o, outs[0]) for o in outs[1:])
