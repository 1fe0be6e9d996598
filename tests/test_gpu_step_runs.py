"""Several steps in one graph launch (small grids) against the same steps one
call at a time and against the host loop: the same bits, whatever the calls'
lengths and the sort interval.  Needs a GB300."""
import numpy as np
import pytest

import synth
from gpu_helpers import by_id

pytestmark = pytest.mark.gpu

SMALL = synth.small_trench(nx=48, ny=40, depth=12, width=10, ppc=20)


def _sim(w, **kw):
    import paper_1610_03918_gb300 as pg
    sim = pg.Sim(w, **kw)
    for s in (0, 1):
        sim.load_particles(s, synth.maxwellian_load(w, s), v_at_t0=True)
    return sim


def _state(sim):
    # (not the kinetic energy: its sums follow the order of the particles, which no two runs share)
    return [by_id(sim.state(s)) for s in (0, 1)] + [sim.phi(), sim.rho(), *sim.efield()]


@pytest.mark.parametrize("w, kw", [
    (SMALL.replace(sort_every=8), {}),
    (SMALL.replace(sort_every=1), {}),
    (SMALL.replace(sort_every=3), dict(warm_start=2)),
    (SMALL.replace(sort_every=100), dict(warm_start=0)),
    (SMALL.replace(sort_every=5, phi_rf_amp=3.0, omega_rf=0.2), {}),
    (SMALL.replace(sort_every=8, recycle=True), {}),
    (synth.periodic_square_64(ppc=8).replace(sort_every=6), {}),
])
def test_runs_of_steps_equal_single_steps(w, kw):
    import paper_1610_03918_gb300 as pg
    a, b, c = _sim(w, **kw), _sim(w, **kw), _sim(w, graphs=False, **kw)
    for n in (16, 16, 2, 2, 5, 5, 9, 9, 1, 23, 23):   # every length twice: the second one is a run
        a.step(n)
        for _ in range(n):
            b.step(1)
        c.step(n)
    ref = _state(a)
    assert all(np.array_equal(x, y) for x, y in zip(_state(b), ref))
    assert all(np.array_equal(x, y) for x, y in zip(_state(c), ref))
    # counted launches: the runs' steps count as single ones
    assert a.timing()["steps"] == b.timing()["steps"] == 111
    # a changed guess captures the runs again
    for s in (a, b):
        assert pg.load_library().pic_set_warm_start(s.ctx, 1 if kw.get("warm_start", 1) != 1 else 2) == pg.PIC_OK
    a.step(8)
    a.step(8)
    for _ in range(16):
        b.step(1)
    assert all(np.array_equal(x, y) for x, y in zip(_state(a), _state(b)))
