"""pic_deposit_static's two scratch layouts and its integer coordinate split,
against the same fixed-point arithmetic restated in numpy: the sums are
integers, so the densities are equal bit for bit.  Needs a GB300."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def restated(nx, ny, px, py, x, y, weight):
    if px:
        x = np.where((x >= 0) & (x < nx), x, np.mod(x, nx))
    if py:
        y = np.where((y >= 0) & (y < ny), y, np.mod(y, ny))
    ok = (x >= 0) & (x < nx) & (y >= 0) & (y < ny)
    x, y = x[ok], y[ok]
    i, j = np.floor(x), np.floor(y)
    lim = np.float32(1 - 2.0 ** -24)
    fx, fy = (np.minimum((a - b).astype(np.float32), lim) for a, b in ((x, i), (y, j)))
    gx, gy, q = np.float32(1) - fx, np.float32(1) - fy, np.float32(2 ** 20)
    w00, w10, w01 = (np.rint((a * b) * q).astype(np.int64) for a, b in ((gx, gy), (fx, gy), (gx, fy)))
    n0, n1 = nx + (not px), ny + (not py)
    acc = np.zeros((n0, n1), np.int64)
    i, j = i.astype(np.int64), j.astype(np.int64)
    for a, b, w in ((0, 0, w00), (1, 0, w10), (0, 1, w01), (1, 1, 2 ** 20 - w00 - w10 - w01)):
        np.add.at(acc, ((i + a) % n0, (j + b) % n1), w)
    return (weight / 2 ** 20) * acc.astype(np.float64)


@pytest.mark.parametrize("nx,ny,px,py,n", [
    (1024, 512, 0, 1, 40000),     # pairs: the scratch exactly full
    (1000, 1000, 0, 1, 40000),    # too large for pairs
    (1000, 1000, 1, 0, 333),
    (37, 29, 1, 1, 5000),
    (5, 7, 0, 0, 1),              # one particle: three lanes of its group of four idle
    (2, 2, 1, 1, 70),             # both neighbours the same node
])
def test_layouts_equal_the_restated_sums(nx, ny, px, py, n):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1610_03918_gb300 as pg
    f = pg.load_library().pic_deposit_static
    f.argtypes = [ctypes.c_int32] * 4 + [ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_double,
                                         ctypes.c_void_p, ctypes.c_void_p]
    f.restype = ctypes.c_int
    rng = np.random.default_rng(n + nx)
    x, y = rng.uniform(-0.01 * nx, 1.01 * nx, n), rng.uniform(-0.01 * ny, 1.01 * ny, n)
    # the edges of the split: zeros, denormals, tiny and nearly whole values, whole ones, the far edge
    edge = [0.0, -0.0, 5e-324, 1e-300, 1e-40, 2.0 ** -60, 2.0 ** -25, 1 - 2.0 ** -53, 1.0, 1 + 2.0 ** -52,
            nx - 2.0 ** -40, float(nx), np.nextafter(float(min(nx, ny)), 0), np.nan, np.inf, -np.inf]
    m = len(edge)
    x = np.concatenate([x, edge, np.full(m, 0.25)])
    y = np.concatenate([y, np.full(m, 0.75), edge])
    with np.errstate(invalid="ignore"):
        ref = restated(nx, ny, px, py, x, y, 0.3)
    xd, yd = (torch.tensor(a, dtype=torch.float64, device="cuda") for a in (x, y))
    for _ in range(2):
        rho = torch.full(ref.shape, float("nan"), dtype=torch.float64, device="cuda")
        st = f(nx, ny, px, py, x.size, xd.data_ptr(), yd.data_ptr(), 0.3, rho.data_ptr(),
               torch.cuda.current_stream().cuda_stream)
        assert st == pg.PIC_OK
        assert np.array_equal(rho.cpu().numpy(), ref)
