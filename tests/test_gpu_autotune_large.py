"""The autotuner on a load of which every tile shape's particles make more chunks than
there are resident CTAs: the tuned run equals one that keeps the 16 x 16 tiles.  Needs
a GB300."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_autotune_on_a_large_load_changes_no_result():
    import paper_1610_03918_gb300 as pg
    w = synth.trench_512x1024(seed=3).replace(ppc=30, sort_every=0)
    parts = [synth.maxwellian_load(w, s) for s in (0, 1)]
    runs = []
    for tune in (True, False):
        sim = pg.Sim(w, capacity=len(parts[0]))
        for s in (0, 1):
            sim.load_particles(s, parts[s], v_at_t0=True)
        sim.step(3)
        if tune:
            assert 0 <= sim.autotune(steps=2) < 4
        else:
            sim.step(4 * 3)
        sim.step(2)
        assert sim.status() == 0
        runs.append([sim.rho(), sim.phi(), *sim.efield(), sim.counts()[0], sim.surface()])
        sim.close()
    assert all(np.array_equal(a, b) for a, b in zip(*runs))
