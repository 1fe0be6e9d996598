"""An ensemble stepped in calls of few steps (one graph of all members), of many (a graph
a group) and timed: the same bits, also where the two kinds alternate.  Needs a GB300."""
import numpy as np
import pytest

import synth
from gpu_helpers import by_id

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 19, 25])
def test_calls_of_any_length_agree(n):
    import paper_1610_03918_gb300 as pg
    ws = [synth.small_trench(nx=32 + 8 * (k % 5), ny=24 + 8 * (k % 3), depth=8, width=4 + k % 4, ppc=4 + k % 3,
                             seed=60 + k).replace(sort_every=5) for k in range(n)]
    loads = [[synth.maxwellian_load(w, s) for s in (0, 1)] for w in ws]
    outs = []
    for calls, timing in (((3, 8, 1, 4, 2, 14), False), ((16, 16), False), ((1,) * 32, False), ((8, 1, 2, 16, 5), True)):
        b = pg.Batch(ws, capacities=[len(p[0]) for p in loads], timing=timing)
        for m, p in zip(b.members, loads):
            for s in (0, 1):
                m.load_particles(s, p[s], v_at_t0=True)
        for steps in calls:
            b.step(steps)
        assert b.timing()["steps"] == (32 if timing else 0)
        outs.append([x for m in b.members for x in (by_id(m.state(0)), by_id(m.state(1)), m.phi(), m.rho(), *m.efield(),
                                                    m.counts()[0], m.surface())])
        b.close()
    for other in outs[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(outs[0], other))
