"""The FP64 pair pass on density sums of exactly zero: mu of a separating pair does
not depend on them."""
import numpy as np
import pytest

import oracle
from gpu_common import jittered, load_state, normwise, oracle_case
from paper_2306_01959_gb300 import sph, workloads as wl

pytestmark = pytest.mark.gpu

TOL = 2e-14  # two roundings of the FP64 sums of a few hundred terms


@pytest.mark.parametrize("kw", [{}, {"delta_mode": sph.DELTA_FULL_SUPPORT}, {"pair_symmetric": 1}])
def test_zero_density_sums_of_separating_pairs(kw):
    c = wl.small_dambreak()
    case = oracle_case(c, **{k: v for k, v in kw.items() if k == "delta_mode"})
    st = jittered(c, seed=12, case=case)
    f = np.flatnonzero(st.type == oracle.FLUID)
    rho = np.full(st.n, 1200.0)  # boundary: no sum with a fluid particle is zero
    rho[f] = 1000.0
    rho[f[::2]] = -1000.0
    u = np.zeros_like(st.u)
    u[f] = 3.0 * (st.r[f] - st.r[f].mean(0))  # every pair of fluid particles separates
    st = oracle.State(st.r, u, rho, st.type)
    sim = sph.Simulation(c, precision=sph.FP64, **kw)
    load_state(sim, st)
    got, ref = sim.derivatives(), oracle.derivatives(case, st)
    assert all(np.all(np.isfinite(ref[k])) for k in range(3))
    assert max(normwise(got[k], ref[k]) for k in range(3)) <= TOL
