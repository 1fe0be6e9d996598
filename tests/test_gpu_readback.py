"""Read-backs that take one wait: node arrays converted on the device in pieces
of the staging buffer, and the layer entry points' error words, one per call in
progress.  Needs a GB300."""
import ctypes
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


# the staging buffer holds 5 values per particle of the capacity: one piece and
# part of the next, many pieces, the x | y seam inside a piece, one value a node more
@pytest.mark.parametrize("capacity", [1, 13, 420, 421, 1 << 16])
def test_node_arrays_in_pieces(capacity):
    import paper_1610_03918_gb300 as pg
    w = synth.small_trench(nx=40, ny=50, depth=12, width=10)
    rho = synth.random_rho(w, seed=3, scale=0.3)
    sim = pg.Sim(w, capacity=capacity)
    sim.set_rho_ext(rho)
    sim.step(0)
    phi, (ex, ey) = sim.phi(), sim.efield()
    assert np.allclose(sim.rho(), rho, rtol=0, atol=1e-12 * np.abs(rho).max())
    ref = pg.Sim(w, capacity=1 << 17)
    ref.set_rho_ext(rho)
    ref.step(0)
    assert np.array_equal(phi, ref.phi())
    assert np.array_equal(np.stack([ex, ey]), np.stack(ref.efield()))
    # interior nodes: the field is the centred difference of the potential, held in FP32
    assert np.abs(ex[1:-1] + 0.5 * (phi[2:] - phi[:-2]))[:20].max() <= 2e-6 * np.abs(ex).max()
    short = np.empty(phi.size - 1)
    st, _ = pg.pic_diag(sim.ctx, pg.PIC_DIAG_PHI, short)
    assert st == pg.PIC_EINVAL


def test_layer_calls_from_several_threads():
    import torch
    import paper_1610_03918_gb300 as pg
    f = pg.load_library().pic_conv3x3_bf16
    f.argtypes = [ctypes.c_int32] * 4 + [ctypes.c_void_p] + [ctypes.c_int32] * 3 + [ctypes.c_void_p] * 2 + \
        [ctypes.c_int32, ctypes.c_void_p] + [ctypes.c_int32] * 3 + [ctypes.c_void_p]
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((1, 40, 136, 32), generator=g, device="cuda").bfloat16()
    w = torch.randn((32, 3, 3, 32), generator=g, device="cuda").bfloat16()
    b = torch.randn((32,), generator=g, device="cuda")
    torch.cuda.synchronize()

    def call(_):
        s = torch.cuda.Stream()
        out = torch.empty((1, 40, 136, 32), dtype=torch.bfloat16, device="cuda")
        s.wait_stream(torch.cuda.current_stream())
        for _ in range(20):
            st = f(0, 1, 40, 136, x.data_ptr(), 32, 0, 32, w.data_ptr(), b.data_ptr(), 1, out.data_ptr(), 32, 0, 32,
                   s.cuda_stream)
            if st != pg.PIC_OK:
                return st, None
        return st, out

    with ThreadPoolExecutor(8) as ex:
        res = list(ex.map(call, range(16)))
    assert all(st == pg.PIC_OK for st, _ in res)
    assert all(torch.equal(o, res[0][1]) for _, o in res)
