"""pic_deposit_static on both sides of the line between its scratch layouts (two sums per
cell row and node column from 8192 particles and half a particle a node on): the sums of
the restated arithmetic, bit for bit.  Needs a GB300."""
import ctypes

import numpy as np
import pytest

from test_gpu_deposit_layouts import restated

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,px,py,n", [
    (1024, 512, 0, 1, 262_399), (1024, 512, 0, 1, 262_400),   # 1025 x 512 nodes; the scratch exactly full
    (1024, 511, 0, 1, 300_000),
    (37, 29, 1, 1, 8191), (37, 29, 1, 1, 8192), (37, 29, 0, 1, 8193),
    (5, 7, 0, 0, 8192), (2, 2, 1, 1, 9001), (1, 40, 1, 0, 10_000), (40, 1, 0, 1, 10_000),
    (1000, 1000, 0, 0, 600_000),                              # no room for pairs
])
def test_layouts_around_the_line(nx, ny, px, py, n):
    import torch
    import paper_1610_03918_gb300 as pg
    f = pg.load_library().pic_deposit_static
    f.argtypes = [ctypes.c_int32] * 4 + [ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_double,
                                         ctypes.c_void_p, ctypes.c_void_p]
    f.restype = ctypes.c_int
    rng = np.random.default_rng(n + nx)
    x, y = rng.uniform(-0.01 * nx, 1.01 * nx, n), rng.uniform(-0.01 * ny, 1.01 * ny, n)
    ref = restated(nx, ny, px, py, x, y, 0.3)
    xd, yd = (torch.tensor(a, dtype=torch.float64, device="cuda") for a in (x, y))
    rho = torch.full(ref.shape, float("nan"), dtype=torch.float64, device="cuda")
    assert f(nx, ny, px, py, n, xd.data_ptr(), yd.data_ptr(), 0.3, rho.data_ptr(),
             torch.cuda.current_stream().cuda_stream) == pg.PIC_OK
    assert np.array_equal(rho.cpu().numpy(), ref)
