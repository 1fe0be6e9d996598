"""The transposed convolution's data gradient with 256 channels on both sides of the
line between its persistent kernel and the tile kernel (K = 1024 from 760 tiles of 128
pixels on, K = 1280 from 380): against the CUDA-core kernel of the same entry point.
Needs a GB300."""
import numpy as np
import pytest

from test_gpu_conv import bf16_round, lib, run_upback  # noqa: F401 (lib: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B, H, W, cin, cout", [
    (3, 253, 128, 256, 256), (3, 254, 128, 256, 256), (1, 380, 128, 256, 320), (1, 381, 120, 256, 320),
])
def test_data_gradient_around_the_line(lib, B, H, W, cin, cout):  # noqa: F811
    rng = np.random.default_rng(H + cout)
    g = bf16_round(rng.standard_normal((B, 2 * H, 2 * W, cout)).astype(np.float32))
    w = bf16_round((rng.standard_normal((2, 2, cin, cout)) / np.sqrt(4 * cout)).astype(np.float32))
    got, st = run_upback(lib, 0, g, 0, cout, w, cin)
    ref, st1 = run_upback(lib, 1, g, 0, cout, w, cin)
    assert st == st1 == lib.PIC_OK
    # both sum in FP32 (K = 4 cout products of order 1 / sqrt(K)) and round to BF16: half
    # a unit in the last place each, a whole one apart at most but for the sums' own error
    assert np.all(np.abs(got - ref) <= 2.0 ** -7 * np.abs(ref) + 1e-5 * np.abs(ref).max())
