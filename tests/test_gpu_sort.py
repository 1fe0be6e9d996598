"""The tile sort: a run that sorts at every step, one that sorts every third
and one that never sorts after the load advance the same particles, bit for bit
(the deposit is in integers, so the order of the particles changes nothing).
Needs a GB300."""
import numpy as np
import pytest

import synth
from gpu_helpers import by_id
from synth import Particles

pytestmark = pytest.mark.gpu


def _load(w, n, seed):
    rng = np.random.default_rng(seed)
    m = synth.plasma_cells(w)
    ci, cj = np.nonzero(m)
    k = rng.integers(0, ci.size, n)
    return Particles(ci[k] + rng.random(n), cj[k] + rng.random(n), 3.0 * rng.standard_normal(n),
                     3.0 * rng.standard_normal(n), np.arange(n, dtype=np.uint32))


FORMS = [
    # workload, particles of each species: fewer than a vector, a unit of the scatter and one more,
    # units of many tiles, species of different sizes, none of one species
    (synth.small_trench(nx=16, ny=16, depth=4, width=4), (1, 3)),
    (synth.small_trench(nx=40, ny=24, depth=8, width=6), (1024, 1025)),
    (synth.small_trench(nx=256, ny=128, depth=0, width=0), (5000, 31)),
    (synth.small_trench(nx=64, ny=32), (70001, 0)),
    (synth.periodic_square_64(), (30000, 50000)),
    (synth.small_trench(nx=1024, ny=512, depth=0, width=0), (60000, 60000)),
    # more tiles than the scatter keeps in shared memory, and than the histogram does
    (synth.small_trench(nx=2176, ny=1024, depth=0, width=0), (30000, 20000)),
    (synth.small_trench(nx=2176, ny=2048, depth=0, width=0), (30000, 20000)),
]


@pytest.mark.parametrize("k", range(len(FORMS)))
def test_sorting_changes_no_particle(k):
    import paper_1610_03918_gb300 as pg
    w, counts = FORMS[k]
    w = w.replace(ppc=400)          # a weak field: what is compared is the motion between tiles
    ref = None
    for every in (1, 3, 1000):
        sim = pg.Sim(w.replace(sort_every=every), capacity=max(counts) + 17, hit_capacity=1 << 17)
        for s in (0, 1):
            if counts[s]:
                sim.load_particles(s, _load(w, counts[s], 100 * k + s), v_at_t0=True)
        sim.step(7)
        got = [by_id(sim.state(s)) for s in (0, 1)] + [sim.rho(), sim.phi()]
        sim.close()
        if ref is None:
            ref = got
            assert got[0].shape[1] + got[1].shape[1] > 0
        else:
            assert all(np.array_equal(a, b) for a, b in zip(got, ref))
