"""The transform solve (csrc/boxpoisson.cu) on every form of box it takes,
against the oracle's sparse direct solve and against the multigrid PCG that
serves the same boxes on request.  Bounds as in the solver tests of
test_gpu_parity.py: relative residual 1e-10 in FP64, potentials within 1e-8
of each other's largest value (both are solved to 1e-10).  Needs a GB300."""
import numpy as np
import pytest

import synth
from oracle import field as ofield
from oracle import poisson as opoisson
from oracle.geometry import from_workload

pytestmark = pytest.mark.gpu

P, B = synth.periodic_square_64, synth.bounded_square_256
FORMS = {
    # slab and slot: ny with odd factors, wide and narrow trenches, a slot of one row
    "trench_30": synth.small_trench(nx=80, ny=30, depth=20, width=15),
    "trench_66_wide": synth.small_trench(nx=40, ny=66, depth=9, width=50),
    "trench_edge_rows": synth.small_trench(nx=12, ny=22, depth=3, width=4),
    # slab alone: plates, a flat electrode, a one-cell trench (its column is all wall)
    "plates_50": synth.small_trench(nx=34, ny=50, depth=0, width=0),
    "flat_slab": synth.small_trench(nx=40, ny=36, depth=10, width=0),
    "trench_one_cell": synth.small_trench(nx=40, ny=36, depth=10, width=1),
    "two_columns": synth.small_trench(nx=16, ny=2, depth=0, width=0),
    # y bounded: odd counts, columns beyond one CTA's 128, a trench, one along the side wall
    "bounded_odd": B(nx=33, ny=27),
    "bounded_wide": B(nx=24, ny=260),
    "bounded_trench": synth.small_trench(nx=40, ny=41, depth=12, width=9).replace(periodic_y=False),
    "bounded_trench_side": synth.small_trench(nx=36, ny=30, depth=8, width=7).replace(periodic_y=False, trench_y0=0),
    # x periodic: doubly periodic (singular), and between two walls in y
    "periodic_36x50": P(nx=36, ny=50),
    "periodic_64": P(),
    "ring_bounded": P(nx=40, ny=31).replace(periodic_y=False),
    # more rows than lanes x runs of one, and than one pass of the solve's warps
    "tall": synth.small_trench(nx=400, ny=12, depth=60, width=4),
}


@pytest.mark.parametrize("name", list(FORMS))
def test_transform_solve_matches_oracle_and_multigrid(name):
    import paper_1610_03918_gb300 as pg
    w = FORMS[name].replace(poisson_rtol=1e-10)
    geom = from_workload(w)
    rho = synth.random_rho(w, seed=31, scale=0.3)
    phis = []
    for method in (pg.POISSON_AUTO, pg.POISSON_MULTIGRID):
        gs = pg.Sim(w, poisson_method=method)
        gs.set_rho_ext(rho)
        gs.step(0)
        assert gs.poisson_stats()[2] <= 1e-10
        phi = gs.phi()
        assert opoisson.residual_rel(geom, phi, rho) <= 2e-10
        phis.append(phi)
        if method == pg.POISSON_AUTO:
            assert gs.poisson_stats()[0] <= 5      # transform passes, not CG iterations
            ex, ey = gs.efield()
            exo, eyo = ofield.efield(geom, opoisson.solve_direct(geom, rho))
            emax = max(np.abs(exo).max(), np.abs(eyo).max())
            assert max(np.abs(ex - exo).max(), np.abs(ey - eyo).max()) <= 1e-5 * emax
        gs.close()
    assert np.abs(phis[0] - phis[1]).max() <= 1e-8 * np.abs(phis[1]).max()
