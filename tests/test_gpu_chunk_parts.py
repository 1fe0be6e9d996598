"""Chunks of more particles than a node's 32-bit sum takes: the density carried
between their parts.  A context of its own makes such chunks of 40M particles, a
member of an ensemble does not; both advance the same particles.  Needs a GB300."""
import numpy as np
import pytest

import synth
from synth import Particles

pytestmark = pytest.mark.gpu

N = 20_000_000     # of each species: 7.3k particles a chunk, two parts


@pytest.mark.parametrize("corner", [True, False])
def test_parts_of_a_chunk(corner):
    import paper_1610_03918_gb300 as pg
    w = synth.bounded_square_256(nx=32, ny=32).replace(ppc=40_000, sort_every=2)
    rng = np.random.default_rng(5)
    loads = []
    for s in (0, 1):
        if corner:   # all next to one node: the largest sums, and on the far nodes many shares of -1
            x, y = (8.0 + np.where(rng.random(N) < 0.5, 1e-5, -1e-5) * rng.random(N) for _ in (0, 1))
        else:
            x, y = (1.0 + 30.0 * rng.random(N) for _ in (0, 1))
        v = 0.05 * rng.standard_normal((2, N))
        loads.append(Particles(x, y, v[0], v[1], np.arange(N, dtype=np.uint32)))
    few = synth.maxwellian_load(w, 0, ppc=2)

    def load(sim, parts):
        for s in (0, 1):
            sim.load_particles(s, parts[s], v_at_t0=True)

    solo = pg.Sim(w, capacity=N)
    load(solo, loads)
    solo.step(3)
    one = [solo.rho(), solo.phi(), *solo.efield(), solo.counts()[1]]
    sums = [solo.state(s)[:4].sum(axis=1) for s in (0, 1)]
    solo.close()
    batch = pg.Batch([w, w], capacities=[N, few.x.size])
    load(batch.members[0], loads)
    load(batch.members[1], [few, few])
    batch.step(3)
    m = batch.members[0]
    other = [m.rho(), m.phi(), *m.efield(), m.counts()[1]]
    assert all(np.array_equal(a, b) for a, b in zip(one, other))
    # the particles themselves: sums over all of them (in any order)
    for s in (0, 1):
        assert np.allclose(m.state(s)[:4].sum(axis=1), sums[s], rtol=1e-10, atol=1e-6)
    batch.close()
