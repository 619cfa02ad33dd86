"""The grid that callers see after autotuning: that of the tuned cell_div by its
definition, whatever grid the pair pass works on."""
import numpy as np
import pytest

import oracle
from gpu_common import oracle_case
from paper_2306_01959_gb300 import sph, workloads as wl

pytestmark = pytest.mark.gpu


# 2h = 0.0831 and 0.06: extents of an odd number of half supports along some axis
# (where twice the cells of 2h are one too many); cells of 2h for callers before the
# tuning
@pytest.mark.parametrize("hfac", [1.2 * 3**0.5, 1.5])
@pytest.mark.parametrize("kw", [{}, {"cell_div": 1}, {"precision": sph.FP64}])
def test_cells_by_definition(hfac, kw):
    dp = 0.02
    c = wl.Case("tuned", (1.03, 0.44, 0.35), (0.4, 0.44, 0.2), None, dp, h=hfac * dp)
    sim = sph.Simulation(c, **{"precision": sph.MIXED, **kw})
    first = 2 if kw.get("precision") == sph.FP64 else 1
    assert sim.tuned_config()["cell_div"] == first
    odd = 0
    for tuned in range(4):
        div = sim.tuned_config()["cell_div"]
        case = oracle_case(c, cell_div=div)
        _, _, dims = oracle.grid_info(case)
        odd += any(d % 2 for d in dims)
        assert sim.n_cells == int(np.prod(dims))
        cell, _, start = sim.cells()
        o_cell, _, o_start = oracle.cells(case, sim.get_state()["r"])
        assert np.array_equal(cell, o_cell) and np.array_equal(start, o_start[:-1])
        sim.step(0.0, 3)
        sim.autotune(2)
    assert odd
