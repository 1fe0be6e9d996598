"""Which small grids end a captured step's solve in the closing cluster (its further
passes are dense transforms on 16 SMs) and which repeat their solver's kernels: seen from
the kernels counted, which follow the passes only in the second case.  Needs a GB300."""
import numpy as np
import pytest

import synth
from gpu_helpers import FIELD_TOL

pytestmark = pytest.mark.gpu

FFT_KERNELS = 4   # of a pass on a grid with a slot


@pytest.mark.parametrize("nx, ny, rtol, warm_start, closed", [
    (64, 64, 1e-10, 1, True),      # few nodes: whatever the passes
    (64, 64, 1e-10, 0, True),
    (168, 128, 1e-10, 1, False),   # just more than those
    (72, 256, 1e-6, 1, True),      # one pass a step
    (72, 256, 1e-6, 2, True),
    (72, 256, 1e-10, 1, False),    # two
    (72, 256, 1e-6, 0, False),
    (440, 64, 1e-6, 1, False),     # more rows than one pass is sure for
    (24, 512, 1e-6, 1, False),     # more columns
])
def test_further_passes_of_fft_grids(nx, ny, rtol, warm_start, closed):
    import paper_1610_03918_gb300 as pg
    w = synth.small_trench(nx=nx, ny=ny, depth=max(3, nx // 5), width=12).replace(poisson_rtol=rtol, ppc=8, sort_every=50)
    sims = [pg.Sim(w, graphs=g, warm_start=warm_start) for g in (True, False)]
    for sim in sims:
        assert sim.solver() == pg.POISSON_AUTO
        for s in (0, 1):
            sim.load_particles(s, synth.maxwellian_load(w, s), v_at_t0=True)
        sim.step(0)
    sim, loop = sims
    sim.timing()
    steps, passes = 6, 0
    for _ in range(steps):
        sim.step(1)
        loop.step(1)
        passes += int(sim.poisson_stats()[1])
        assert sim.poisson_stats()[2] <= rtol
    t = sim.timing()
    # the particle kernel, the guess (0: two kernels and the density; 2: two, the density), the solve
    fixed = 1 + (0 if warm_start == 1 else 3) + 1
    expected = steps * (fixed + 1 + FFT_KERNELS) if closed else steps * fixed + passes * (1 + FFT_KERNELS)
    assert t["steps"] == steps and t["launches"] == expected + 3 * t["sorts"]
    E, El = np.stack(sim.efield()), np.stack(loop.efield())
    assert np.abs(E - El).max() <= max(FIELD_TOL, 100 * rtol) * np.abs(El).max()
    for sim in sims:
        sim.close()


@pytest.mark.parametrize("nx, ny, closed", [(24, 513, True), (24, 514, False), (16, 512, True)])
def test_further_passes_of_boxes(nx, ny, closed):
    # between four walls: ny - 1 columns, two kernels a pass
    import paper_1610_03918_gb300 as pg
    w = synth.bounded_square_256(nx=nx, ny=ny).replace(poisson_rtol=1e-10, ppc=8, sort_every=50)
    sims = [pg.Sim(w, graphs=g) for g in (True, False)]
    for sim in sims:
        for s in (0, 1):
            sim.load_particles(s, synth.maxwellian_load(w, s), v_at_t0=True)
        sim.step(0)
    sim, loop = sims
    sim.timing()
    steps, passes = 6, 0
    for _ in range(steps):
        sim.step(1)
        loop.step(1)
        passes += int(sim.poisson_stats()[1])
        assert sim.poisson_stats()[2] <= 1e-10
    t = sim.timing()
    assert passes > steps
    expected = steps * (2 + 1 + 2) if closed else 2 * steps + passes * (1 + 2)
    assert t["steps"] == steps and t["launches"] == expected + 3 * t["sorts"]
    E, El = np.stack(sim.efield()), np.stack(loop.efield())
    assert np.abs(E - El).max() <= FIELD_TOL * np.abs(El).max()
    for sim in sims:
        sim.close()
