"""The FP64 pair pass on fixed-point positions against the oracle, and against the
same pass on doubles, which takes over for tanks longer than 512 supports."""
import dataclasses

import numpy as np
import pytest

import oracle
from gpu_common import jittered, load_state, normwise, oracle_case
from paper_2306_01959_gb300 import sph, workloads as wl

pytestmark = pytest.mark.gpu

# two roundings of the FP64 sums of a few hundred terms
TOL = 2e-14


def _derivatives(c, r, u, rho, types, **kw):
    sim = sph.Simulation(c, precision=sph.FP64, **kw)
    load_state(sim, oracle.State(r, u, rho, types))
    return sim.derivatives()


# 2h just below, at and above a power of two (the fixed-point unit changes there),
# other scales of length, both readings of the delta term, each pair once
@pytest.mark.parametrize("scale", [1.0, 0.0625 / 0.0831384, 0.0625 / 0.0831384 * (1 + 1e-15), 1e-3, 37.0])
@pytest.mark.parametrize("kw", [{}, {"delta_mode": sph.DELTA_FULL_SUPPORT}, {"pair_symmetric": 1}])
def test_fixed_point_matches_oracle_at_every_scale(scale, kw):
    dp = 0.02 * scale
    c = wl.Case("fixed", tuple(scale * v for v in (0.6, 0.3, 0.4)), tuple(scale * v for v in (0.4, 0.3, 0.26)), None, dp)
    case = oracle_case(c, **{k: v for k, v in kw.items() if k == "delta_mode"})
    st = jittered(c, seed=11, case=case)
    got, ref = _derivatives(c, st.r, st.u, st.rho, st.type, **kw), oracle.derivatives(case, st)
    err = [normwise(got[k], ref[k]) for k in range(3)]
    assert max(err) <= TOL and np.array_equal(got[3], ref[3]), err


def test_near_pairs_and_coincident_particles():
    # pairs from 2h / 16 down to 0, across the distance below which the FP64
    # operations replace the integer ones
    c = wl.small_dambreak()
    case = oracle_case(c)
    st = jittered(c, seed=2, case=case)
    f = np.flatnonzero(st.type == oracle.FLUID)
    r = st.r.copy()
    rng = np.random.Generator(np.random.PCG64(4))
    for k, gap in enumerate([2.0**-m for m in range(4, 24)] + [1e-12, 0.0]):
        d = rng.normal(size=3)
        r[f[2 * k + 1]] = r[f[2 * k]] + d / np.linalg.norm(d) * gap * 2.0 * c.h
    st = oracle.State(r, st.u, st.rho, st.type)
    got, ref = _derivatives(c, st.r, st.u, st.rho, st.type), oracle.derivatives(case, st)
    assert max(normwise(got[k], ref[k]) for k in range(3)) <= TOL
    assert np.array_equal(got[3], ref[3])


def test_long_tank_takes_the_double_positions():
    # the same column in a tank of 515 supports and in one of 500
    out = []
    for length in (515.0, 500.0):
        h = 0.024
        c = wl.Case("long", (2 * h * length, 0.08, 0.1), (0.2, 0.08, 0.06), None, 0.02, h=h)
        case = oracle_case(c)
        st = jittered(c, seed=6, case=case)
        nf = int((st.type == oracle.FLUID).sum())
        got, ref = _derivatives(c, st.r, st.u, st.rho, st.type), oracle.derivatives(case, st)
        assert max(normwise(got[k], ref[k]) for k in range(3)) <= TOL
        assert np.array_equal(got[3], ref[3])
        out.append([g[:nf] for g in got])
    assert not np.array_equal(out[0][1], out[1][1])  # two different paths


# 9, 25 and 49 rows of cells: up to two loads of row ranges by the 32 lanes, and
# rows that are empty or outside the grid (the column fills a part of the tank)
@pytest.mark.parametrize("cell_div", [1, 2, 3])
@pytest.mark.parametrize("kw", [{}, {"pair_symmetric": 1}])
def test_rows_of_every_cell_size(cell_div, kw):
    c = wl.small_dambreak()
    case = oracle_case(c)
    st = jittered(c, seed=5, case=case)
    got, ref = _derivatives(c, st.r, st.u, st.rho, st.type, cell_div=cell_div, **kw), oracle.derivatives(case, st)
    assert max(normwise(got[k], ref[k]) for k in range(3)) <= TOL
    assert np.array_equal(got[3], ref[3])


def test_density_sums_that_are_not_positive():
    # rho_i + rho_j negative, or positive from two signs: the integer reciprocal
    # leaves the former to the FP64 operations
    c = wl.small_dambreak()
    case = oracle_case(c)
    st = jittered(c, seed=8, case=case)
    rho = st.rho.copy()
    f = np.flatnonzero(st.type == oracle.FLUID)
    rho[f[::3]] *= -1.3
    got = _derivatives(c, st.r, st.u, rho, st.type)
    ref = oracle.derivatives(case, oracle.State(st.r, st.u, rho, st.type))
    assert max(normwise(got[k], ref[k]) for k in range(3)) <= TOL
    assert np.array_equal(got[3], ref[3])
