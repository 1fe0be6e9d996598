"""A captured step whose solve cannot reach its tolerance: the small grids' closing
cluster stops after its pass cap, sets PIC_ST_NOCONV and leaves the field it has.  (The
host loop's step returns the same as its status.)  The load is neutral at every node, so
its own solve (of 0) succeeds and the steps are the first to give up.  Needs a GB300."""
import numpy as np
import pytest

import synth
from gpu_helpers import FIELD_TOL
from synth import Particles

pytestmark = pytest.mark.gpu

BOXES = {
    "transform": synth.bounded_square_256(nx=32, ny=32),
    "fft": synth.small_trench(nx=32, ny=32, depth=0, width=0).replace(phi_electrode=0.0),
    "slot": synth.small_trench(nx=40, ny=30, depth=10, width=8).replace(phi_electrode=0.0, surface_charge=False),
    "singular": synth.periodic_square_64(nx=32, ny=32),
}
MAX_PASSES = 8   # of a solve


def _run(w, rtol):
    import paper_1610_03918_gb300 as pg
    sim = pg.Sim(w.replace(poisson_rtol=rtol))
    e = synth.maxwellian_load(w, 0)
    for s in (0, 1):   # the ions start where the electrons do
        sim.load_particles(s, e if s == 0 else Particles(e.x, e.y, 0.0 * e.vx, 0.0 * e.vy, e.ids), v_at_t0=True)
    sim.step(0)
    assert sim.status() == 0
    sim.step(1)
    return sim


@pytest.mark.parametrize("name", list(BOXES))
def test_unreachable_tolerance_in_a_step(name):
    import paper_1610_03918_gb300 as pg
    w = BOXES[name].replace(ppc=8, sort_every=4)
    sim, ref = _run(w, 1e-30), _run(w, 1e-10)
    assert sim.status() == pg.PIC_ST_NOCONV and ref.status() == 0   # (reading clears it)
    assert sim.poisson_stats()[1] == MAX_PASSES and ref.poisson_stats()[1] < MAX_PASSES
    E, Er = np.stack(sim.efield()), np.stack(ref.efield())
    assert np.abs(E - Er).max() <= FIELD_TOL * np.abs(Er).max()
    for _ in range(4):   # single steps, then runs of them
        sim.step(4)
        assert sim.status() == pg.PIC_ST_NOCONV
        assert sim.poisson_stats()[1] == MAX_PASSES
    sim.close()
    ref.close()
