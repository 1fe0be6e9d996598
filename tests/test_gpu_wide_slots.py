"""The FFT solve on trenches of 110 columns and more, whose sine basis takes more shared
memory than a kernel has without asking: against the oracle's sparse direct solve, in
the host loop and in captured steps.  Bounds as in test_gpu_box_solver.py.  Needs a
GB300."""
import numpy as np
import pytest

import synth
from gpu_helpers import FIELD_TOL
from oracle import field as ofield
from oracle import poisson as opoisson
from oracle.geometry import from_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny, width", [(128, 110), (128, 111), (128, 120), (256, 150), (256, 160), (256, 161), (512, 140)])
def test_wide_slots(ny, width):
    # width cells: width - 1 columns between the walls; from 160 columns on the box solver's
    import paper_1610_03918_gb300 as pg
    w = synth.small_trench(nx=40, ny=ny, depth=14, width=width).replace(poisson_rtol=1e-10)
    geom = from_workload(w)
    rho = synth.random_rho(w, seed=8, scale=0.3)
    sim = pg.Sim(w, capacity=16)
    assert sim.solver() == (pg.POISSON_AUTO if width <= 160 else pg.POISSON_MULTIGRID)
    sim.set_rho_ext(rho)
    sim.step(0)
    assert opoisson.residual_rel(geom, sim.phi(), rho) <= 2e-10
    exo, eyo = ofield.efield(geom, opoisson.solve_direct(geom, rho))
    for _ in range(2):   # the second time after captured steps of the same density
        ex, ey = sim.efield()
        emax = max(np.abs(exo).max(), np.abs(eyo).max())
        assert max(np.abs(ex - exo).max(), np.abs(ey - eyo).max()) <= FIELD_TOL * emax
        sim.step(3)
        assert sim.status() == 0 and sim.poisson_stats()[2] <= 1e-10
    sim.close()
