"""The cell size of the tiled mixed pass: cells of h, or of 2h where h < 1.75 dp (the
automatic size: below 48,000 particles), while callers see cells of 2h."""
import numpy as np
import pytest

import oracle
from gpu_common import jittered, load_state, normwise, oracle_case
from paper_2306_01959_gb300 import sph, workloads as wl

pytestmark = pytest.mark.gpu

TOL = 5e-6        # the bar of test_gpu_pair_tiles
MIXED_TOL = 2e-4  # of the clumped states in test_gpu_parity


def _check(c, kw, st, tol):
    case = oracle_case(c)
    sim = sph.Simulation(c, precision=sph.MIXED, **kw)
    load_state(sim, st)
    got, ref = sim.derivatives(), oracle.derivatives(case, st)
    err = [normwise(got[k], ref[k]) for k in range(3)]
    assert max(err) <= tol, err
    f = st.type == oracle.FLUID  # (a pair within one FP32 rounding of 2h may fall on either side)
    assert np.abs(got[3] - ref[3])[f].max() <= 2 and (got[3] != ref[3])[f].sum() <= 40
    cell, _, start = sim.cells()
    o_cell, _, o_start = oracle.cells(oracle_case(c, cell_div=1), sim.get_state()["r"])
    assert np.array_equal(cell, o_cell) and np.array_equal(start, o_start[:-1])
    assert sim.tuned_config()["cell_div"] == 1
    sim.sync()


# both sides of the line in h / dp, and of the one in particles (18,532 and 51,750)
@pytest.mark.parametrize("hfac", [1.0, 1.5, 1.749, 1.75, 2.3])
@pytest.mark.parametrize("dp", [0.02, 0.0131])
@pytest.mark.parametrize("kw", [{}, {"cell_div": 1}, {"pair_group": 2}])
def test_both_sides_match_oracle(hfac, dp, kw):
    c = wl.Case("cells", (1.0, 0.5, 0.5), (0.4, 0.5, 0.3), None, dp, h=hfac * dp)
    _check(c, kw, jittered(c, seed=int(100 * hfac), case=oracle_case(c)), TOL)


# compressed fluid: tiles of cells of 2h are halved down to one, and read from global memory
@pytest.mark.parametrize("factor", [0.85, 0.7, 0.5, 0.35])
@pytest.mark.parametrize("kw", [{}, {"cell_div": 1, "delta_mode": sph.DELTA_ALL_FLUID}])
def test_compressed_with_cells_of_two_h(factor, kw):
    dp = 0.0171
    c = wl.Case("cells", (0.62, 0.33, 0.41), (0.4, 0.33, 0.25), None, dp, h=1.5 * dp)
    st = jittered(c, seed=9, case=oracle_case(c))
    r = st.r.copy()
    r[st.type == oracle.FLUID] *= factor
    _check(c, kw, oracle.State(r, st.u, st.rho, st.type), MIXED_TOL)


def test_batch_takes_one_size():
    # instances on either side of the line: the same results as each for itself, to rounding
    dp = 0.02
    cases = [wl.Case(f"b{k}", (0.7, 0.4, 0.4), (0.3, 0.4, 0.2), None, dp, h=f * dp) for k, f in enumerate((1.4, 2.0))]
    b = sph.Simulation(cases, precision=sph.MIXED, batch=True)
    b.step(1e-4, 20)
    s = b.get_state()
    at = 0
    for c in cases:
        one = sph.Simulation(c, precision=sph.MIXED)
        one.step(1e-4, 20)
        g = one.get_state()
        for k, tol in (("r", 1e-8), ("u", 2e-5), ("rho", 1e-2)):
            assert np.abs(s[k][at : at + one.n] - g[k]).max() <= tol, k
        at += one.n
    assert at == b.n
