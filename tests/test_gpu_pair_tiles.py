"""The mixed pair kernel over its tile shapes: spacings and smoothing lengths that
give every kind of tile (large, of cell_div cells, smaller, staged in chunks), each
cell size and launch shape, and states its staged path must not take."""
import numpy as np
import pytest

import oracle
from gpu_common import jittered, load_state, normwise, oracle_case
from paper_2306_01959_gb300 import sph, workloads as wl

pytestmark = pytest.mark.gpu

# FP32 offsets and pair terms: about 6e-8 relative per operation, tens of
# operations and a few hundred terms per sum (the bar of test_gpu_parity_more)
TOL = 5e-6


def _case(dp, hfac, tank=(0.62, 0.33, 0.41)):
    """A ragged tank, two thirds full."""
    return wl.Case("tiles", tank, (0.4, tank[1], 0.25), None, dp, h=hfac * dp)


def _errors(sim, st, case):
    got, ref = sim.derivatives(), oracle.derivatives(case, st)
    assert np.array_equal(np.isfinite(got[1]), np.isfinite(ref[1]))
    # counts of the jittered particles only: at h = 1.5 dp and 2.5 dp the boundary
    # lattice has pairs exactly at 2h, which FP32 puts on either side
    nn = np.abs(got[3] - ref[3])[st.type == oracle.FLUID]
    return [normwise(got[k], ref[k]) for k in range(3)], int((nn > 0).sum()), int(nn.max())


# h / dp: sparse cells, the paper's, the workloads', cells that take smaller tiles
# (2.3, 2.5) and neighbourhoods staged in chunks (2.75, 3.4)
@pytest.mark.parametrize("hfac", [0.8, 1.5, 2.078, 2.3, 2.5, 2.75, 3.4])
@pytest.mark.parametrize("delta_mode", [sph.DELTA_ALL_FLUID, sph.DELTA_FULL_SUPPORT])
def test_tile_shapes_match_oracle(hfac, delta_mode):
    c = _case(0.0211, hfac)
    case = oracle_case(c, delta_mode=delta_mode)
    st = jittered(c, seed=int(hfac * 100), case=case, out_of_domain=3)
    sim = sph.Simulation(c, precision=sph.MIXED, delta_mode=delta_mode)
    load_state(sim, st)
    err, differing, most = _errors(sim, st, case)
    assert max(err) <= TOL, err
    # a pair within one FP32 rounding of 2h may fall on either side
    assert most <= 1 and differing <= 8, (differing, most)


@pytest.mark.parametrize("cell_div", [0, 1, 2, 3])
@pytest.mark.parametrize("warps,group", [(8, 4), (8, 2), (16, 4)])
def test_cell_sizes_and_launch_shapes(cell_div, warps, group):
    c = _case(0.0233, 1.9)
    case = oracle_case(c)
    st = jittered(c, seed=3, case=case)
    sim = sph.Simulation(c, precision=sph.MIXED, cell_div=cell_div, pair_warps=warps, pair_group=group)
    load_state(sim, st)
    err, differing, most = _errors(sim, st, case)
    assert max(err) <= TOL and most <= 1 and differing <= 8, (err, differing, most)
    s = sim.pair_stats()
    o = oracle.derivatives(case, st)
    assert abs(s["in_support"] - int(o[3][o[3] >= 0].sum())) <= 8


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e20])
def test_values_a_zero_weight_cannot_cancel_stay_local(value):
    # one particle with such a velocity: the particles beyond 2h of it, some of
    # them sharing clusters and tiles with its neighbours, keep their derivatives
    c = _case(0.0233, 2.078)
    case = oracle_case(c)
    st = jittered(c, seed=5, case=case)
    f = np.flatnonzero(st.type == oracle.FLUID)
    i = f[len(f) // 2]
    sim = sph.Simulation(c, precision=sph.MIXED)
    load_state(sim, st)
    ref = sim.derivatives()
    u = st.u.copy()
    u[i, 0] = value
    load_state(sim, oracle.State(st.r, u, st.rho, st.type))
    got = sim.derivatives()
    # half a percent of room for the FP32 distances
    far = np.linalg.norm(st.r - st.r[i], axis=1) > 2.01 * c.h
    near = ~far & (st.type == oracle.FLUID)
    assert far.sum() > 1000 and near.sum() > 100
    assert np.all(np.isfinite(got[0][far])) and np.all(np.isfinite(got[1][far]))
    assert normwise(got[0][far], ref[0][far]) <= TOL and normwise(got[1][far], ref[1][far]) <= TOL
    assert normwise(got[0][near], ref[0][near]) > 1.0 or not np.all(np.isfinite(got[0][near]))


def test_public_grid_is_the_chosen_one():
    # the automatic cell size is 2h for callers whatever the pair pass works on;
    # reading the cells leaves the run as it was
    c = _case(0.0233, 2.078)
    case = oracle_case(c, cell_div=1)
    a, b = (sph.Simulation(c, precision=sph.MIXED) for _ in range(2))
    st = jittered(c, seed=9, case=case, out_of_domain=2)
    for sim in (a, b):
        load_state(sim, st)
        sim.step(0.0, 5)
    lo, size, dims = oracle.grid_info(case)
    assert a.n_cells == int(np.prod(dims))
    cell, srt, start = a.cells()
    o_cell, _, o_start = oracle.cells(case, a.get_state()["r"])
    assert np.array_equal(cell, o_cell) and np.array_equal(start, o_start[:-1])
    a.step(0.0, 20)
    b.step(0.0, 20)
    sa, sb = a.get_state(), b.get_state()
    assert np.array_equal(sa["r"], sb["r"]) and np.array_equal(sa["rho"], sb["rho"])
