"""Cells of the mixed form on the undisturbed lattice, whose planes lie on cell faces
for some smoothing lengths: the grid's definition (x - lo) / cs decides, after
creation, after a load and after steps."""
import numpy as np
import pytest

import oracle
from gpu_common import oracle_case
from paper_2306_01959_gb300 import sph, workloads as wl

pytestmark = pytest.mark.gpu


def _check(sim, case):
    cell, _, start = sim.cells()
    o_cell, _, o_start = oracle.cells(case, sim.get_state()["r"])
    assert np.array_equal(cell, o_cell) and np.array_equal(start, o_start[:-1])


# h / dp with whole lattice planes where the product with 1/cs rounds to the other cell
# (0.75 and 1.25, 1.75), without any (1.2 sqrt 3), and beyond the tiled pass (2.75)
@pytest.mark.parametrize("hfac", [0.75, 1.25, 1.75, 1.2 * 3**0.5, 2.75])
@pytest.mark.parametrize("cell_div", [0, 1, 2, 3])
def test_lattice_planes_on_faces(hfac, cell_div):
    dp = 0.01
    c = wl.Case("faces", (3.2, 0.08, 0.1), (0.3, 0.08, 0.06), None, dp, h=hfac * dp)
    case = oracle_case(c, cell_div=max(cell_div, 1))
    sim = sph.Simulation(c, precision=sph.MIXED, cell_div=cell_div)
    _check(sim, case)
    sim.restore(sim.checkpoint())
    _check(sim, case)
    sim.step(0.0, 3)
    _check(sim, case)


def test_coordinates_next_to_faces():
    # fluid at and around faces by up to a few roundings, and outside the grid
    dp = 0.01
    c = wl.Case("faces", (0.4, 0.3, 0.3), (0.3, 0.3, 0.2), None, dp, h=1.3 * dp)
    case = oracle_case(c, cell_div=1)
    sim = sph.Simulation(c, precision=sph.MIXED)
    s = sim.get_state()
    lo, size, dims = oracle.grid_info(case)
    lo, dims, cs = np.asarray(lo), np.asarray(dims), float(np.ravel(size)[0])
    rng = np.random.Generator(np.random.PCG64(36))
    f = np.flatnonzero(s["type"] == oracle.FLUID)
    r = s["r"].copy()
    face = lo + rng.integers(-1, dims + 2, (len(f), 3)) * cs * 0.5 ** rng.integers(0, 2, (len(f), 1))
    ulps = rng.integers(-3, 4, (len(f), 3))
    off = np.where(rng.random((len(f), 1)) < 0.5, ulps * np.spacing(np.abs(face)), rng.normal(0, 2e-5 * cs, (len(f), 3)))
    r[f] = face + off
    r[f[0]] = (1e300, 0.1, 0.1)
    r[f[1]] = (0.1, -1e9, 0.1)
    r[f[2]] = (0.1, 0.1, 65536 * cs)
    sim.set_state(r, s["u"], s["rho"])
    _check(sim, case)
