"""Which solver a large box gets: the transform solve takes one to three passes, the
multigrid PCG five iterations and more.  Both meet the tolerance.  Needs a GB300."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box, nx, ny, transform", [
    ("walls", 1024, 1024, True),
    ("walls", 1216, 1024, True),         # multigrid sweeps 19 x 16 cells at its coarsest here
    ("walls", 1536, 1024, False),
    ("walls", 2048, 768, True),          # both sides of the line: 1.20e9 of 1.24e9,
    ("walls", 2176, 768, False),         # 1.28e9 of 1.25e9
    ("ring", 1536, 1024, False),
    ("periodic", 1536, 1024, True),
    ("periodic", 2048, 1024, False),
    ("periodic", 2048, 992, True),       # 64 x 62 cells
])
def test_solver_of_a_large_box(box, nx, ny, transform):
    import paper_1610_03918_gb300 as pg
    w = (synth.bounded_square_256(nx=nx, ny=ny) if box == "walls" else
         synth.periodic_square_64(nx=nx, ny=ny).replace(periodic_y=box == "periodic")).replace(ppc=1)
    sim = pg.Sim(w, capacity=16)
    sim.set_rho_ext(synth.random_rho(w, seed=4, scale=0.3))
    sim.step(0)
    it, _, rel = sim.poisson_stats()[:3]
    sim.close()
    assert rel <= 1e-6
    assert (it <= 3) == transform
