"""The MPS neighbour passes over per-particle lists against the warp-per-particle
ones that take over when a list would be longer than row_width, and the limits of
the one-launch CG solve."""
import numpy as np
import pytest

from gpu_common import normwise
from paper_2306_01959_gb300 import mps, sph

pytestmark = pytest.mark.gpu

L0 = 0.02


def _tank(width, layers=2, nx=13, ny=7, **kw):
    """A shallow pool: a floor particle has 32 particles within r_e, 10 of them
    dummies, a fluid one at most 30 with a pressure."""
    return mps.Tank(((nx + 5) * L0, ny * L0, 0.2), (nx * L0, ny * L0, layers * L0), L0, 3e-4, row_width=width, **kw)


# ragged counts around the 32 rows that share a block of the matrix
@pytest.mark.parametrize("nx,ny", [(13, 7), (8, 4), (16, 16), (31, 9)])
def test_lists_equal_the_search(nx, ny):
    out = []
    for width in (64, 31):  # 31: a floor particle's list does not fit, every row does
        t = _tank(width, nx=nx, ny=ny)
        s = t.get_state()
        rng = np.random.Generator(np.random.PCG64(nx))
        u = np.where((s["type"] == mps.FLUID)[:, None], rng.normal(0.0, 0.05, s["r"].shape), 0.0)
        t.set_state(s["r"], u)
        p = t.pressure()
        size = t.system_size()
        t.step(3)
        out.append((p, size, t.get_state()))
    (pa, na, a), (pb, nb, b) = out
    assert na == nb and np.array_equal(pa["surf"], pb["surf"]) and pa["iterations"] == pb["iterations"]
    # sums of the same terms in another order (and one rounding of 1/r each)
    assert normwise(pa["nd"], pb["nd"]) <= 1e-14 and normwise(pa["P"], pb["P"]) <= 1e-9
    assert normwise(a["r"], b["r"]) <= 1e-12 and normwise(a["u"], b["u"]) <= 1e-9


def test_row_wider_than_its_storage_is_refused():
    t = _tank(24, layers=6)
    with pytest.raises(sph.SphError) as e:
        t.pressure()
    assert e.value.code == sph.SPH_ESTATE


def test_solve_that_does_not_converge_is_reported():
    t = _tank(64, layers=6, cg_max=1, cg_tol=1e-14)
    with pytest.raises(sph.SphError) as e:
        t.step(1)
    assert e.value.code == sph.SPH_EUNSTABLE


def test_zero_right_hand_side_needs_no_iteration():
    # kappa_r = 0: no source anywhere
    t = _tank(64, layers=6, kappa_r=0.0)
    p = t.pressure()
    assert p["iterations"] == 0 and not p["P"].any()
