"""Work counts of a pair pass: the pairs evaluated are those with a fluid particle."""
import numpy as np
import pytest

import oracle
from gpu_common import jittered, load_state, oracle_case
from paper_2306_01959_gb300 import sph, workloads as wl

pytestmark = pytest.mark.gpu


# the tiled pass, the chunked one (h = 2.75 dp) and the FP64 pass
@pytest.mark.parametrize("hfac,kw", [(2.078, {}), (2.078, {"pair_group": 2}), (2.75, {}), (2.75, {"pair_group": 1}),
                                     (2.078, {"precision": sph.FP64})])
def test_evaluated_pairs(hfac, kw):
    dp = 0.0233
    c = wl.Case("stats", (0.62, 0.33, 0.41), (0.4, 0.33, 0.25), None, dp, h=hfac * dp)
    case = oracle_case(c)
    st = jittered(c, seed=4, case=case)
    sim = sph.Simulation(c, **{"precision": sph.MIXED, **kw})
    load_state(sim, st)
    s = sim.pair_stats()
    fluid = st.type == oracle.FLUID
    near = -fluid.astype(np.int64)  # fluid neighbours of every particle
    for p in st.r[fluid]:
        near += ((st.r - p) ** 2).sum(1) < (2.0 * c.h) ** 2
    both = int(oracle.neighbour_counts(case, st.r)[fluid].sum())  # all neighbours of the fluid ones
    # a pair within one FP32 rounding of 2h may fall on either side
    assert abs(s["evaluated"] - (both + int(near[~fluid].sum()))) <= 8
    if s["fluid_fluid"] >= 0:  # (not counted by the FP64 form)
        assert abs(s["fluid_fluid"] - int(near[fluid].sum())) <= 8
