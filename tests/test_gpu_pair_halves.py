"""Compressed states: tiles whose neighbourhood exceeds the staging buffer are halved
until their parts fit, down to single cells, and beyond those read from global memory."""
import numpy as np
import pytest
from scipy import spatial

import oracle
from gpu_common import jittered, load_state, normwise, oracle_case
from paper_2306_01959_gb300 import sph, workloads as wl

pytestmark = pytest.mark.gpu

MIXED_TOL = 2e-4  # the bar of the clumped states in test_gpu_parity


def _squeezed(c, factor, seed, **kw):
    """A jittered state with the fluid compressed towards one corner of the tank."""
    st = jittered(c, seed=seed, case=oracle_case(c, **kw))
    r = st.r.copy()
    f = st.type == oracle.FLUID
    r[f] = np.asarray(c.column) * 0.4 + (r[f] - np.asarray(c.column) * 0.4) * np.asarray(factor)
    return oracle.State(r, st.u, st.rho, st.type)


# compressed evenly (1.2 to 16 times as dense) and along one axis, in a ragged tank
# whose last tiles reach beyond the grid
@pytest.mark.parametrize("factor", [(0.94,) * 3, (0.85,) * 3, (0.7,) * 3, (0.4,) * 3, (1, 1, 0.3), (0.3, 1, 1), (1, 0.4, 0.9)])
@pytest.mark.parametrize("kw", [{}, {"cell_div": 1}, {"cell_div": 3, "pair_group": 2}, {"delta_mode": sph.DELTA_FULL_SUPPORT}])
def test_halved_tiles_match_oracle(factor, kw):
    dp = 0.0171
    c = wl.Case("halves", (0.62, 0.33, 0.41), (0.4, 0.33, 0.25), None, dp, h=2.078 * dp)
    okw = {k: v for k, v in kw.items() if k == "delta_mode"}
    st = _squeezed(c, factor, 5, **okw)
    sim = sph.Simulation(c, precision=sph.MIXED, **kw)
    load_state(sim, st)
    got, ref = sim.derivatives(), oracle.derivatives(oracle_case(c, **okw), st)
    err = [normwise(got[k], ref[k]) for k in range(3)]
    assert max(err) <= MIXED_TOL, err
    f = st.type == oracle.FLUID  # (a pair within one FP32 rounding of 2h may fall on either side)
    assert np.abs(got[3] - ref[3])[f].max() <= 2 and (got[3] != ref[3])[f].sum() <= 40
    sim.sync()


@pytest.mark.parametrize("hfac", [1.5, 2.3])
def test_larger_tiles(hfac):
    # enough particles for tiles of several supports, a clump in a part of them
    dp = 0.01
    c = wl.Case("halves", (1.0, 0.5, 0.5), (0.6, 0.5, 0.3), None, dp, h=hfac * dp)
    case = oracle_case(c)
    st = _squeezed(c, (0.8, 0.9, 0.8), 6)
    sim = sph.Simulation(c, precision=sph.MIXED)
    load_state(sim, st)
    got, ref = sim.derivatives(), oracle.derivatives(case, st)
    err = [normwise(got[k], ref[k]) for k in range(3)]
    assert max(err) <= MIXED_TOL, err
    s = sim.pair_stats()
    # pairs within one FP32 rounding of 2h may fall on either side: at h = 1.5 dp all
    # pairs of the boundary lattice that are 3 dp apart, elsewhere next to none
    tree = spatial.cKDTree(st.r)
    ties = int(tree.count_neighbors(tree, 2 * c.h * (1 + 1e-6)) - tree.count_neighbors(tree, 2 * c.h * (1 - 1e-6)))
    assert abs(s["in_support"] - int(ref[3][ref[3] >= 0].sum())) <= ties


def test_persistent_launch_equals_per_phase():
    dp = 0.0171
    c = wl.Case("halves", (0.62, 0.33, 0.41), (0.4, 0.33, 0.25), None, dp, h=2.078 * dp)
    st = _squeezed(c, (0.8,) * 3, 7)
    out = []
    for kw in ({"persistent": 1}, {"use_graph": 0}, {}):
        sim = sph.Simulation(c, precision=sph.MIXED, **kw)
        load_state(sim, st)
        sim.step(1e-7, 4)
        sim.sync()
        out.append(sim.get_state())
    for k in ("r", "u", "rho"):
        assert np.array_equal(out[0][k], out[1][k]) and np.array_equal(out[0][k], out[2][k]), k


def test_values_that_a_zero_weight_does_not_cancel():
    # a NaN density in a halved tile: its part takes the masked path
    dp = 0.0171
    c = wl.Case("halves", (0.62, 0.33, 0.41), (0.4, 0.33, 0.25), None, dp, h=2.078 * dp)
    case = oracle_case(c)
    st = _squeezed(c, (0.8,) * 3, 8)
    rho = st.rho.copy()
    rho[np.flatnonzero(st.type == oracle.FLUID)[100]] = np.nan
    st = oracle.State(st.r, st.u, rho, st.type)
    sim = sph.Simulation(c, precision=sph.MIXED)
    load_state(sim, st)
    got, ref = sim.derivatives(), oracle.derivatives(case, st)
    ok = np.isfinite(ref[1]).all(1)
    assert np.array_equal(np.isfinite(got[1]).all(1), ok) and not ok.all() and ok.any()
    assert normwise(got[1][ok], ref[1][ok]) <= MIXED_TOL
