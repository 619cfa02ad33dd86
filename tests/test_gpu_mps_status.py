"""Failed MPS steps: the bounded waits of the CG solve, and the handle after a
failure once a state is loaded."""
import numpy as np
import pytest

from paper_2306_01959_gb300 import mps, sph

pytestmark = pytest.mark.gpu

L0 = 0.02


def test_solve_wait_runs_out_and_reports_timeout():
    # one poll per wait: a CTA that arrives early gives up, the others run out at
    # their next barrier, the launch ends and the context stays usable
    args = ((1.0, 0.5, 0.5), (0.4, 0.5, 0.3), L0, 8e-4)
    t = mps.Tank(*args, spin_limit=1)
    with pytest.raises(sph.SphError) as e:
        t.step(1)
    assert e.value.code == sph.SPH_ETIMEOUT
    t.close()
    ok = mps.Tank(*args)
    ok.step(1)
    assert ok.last_solve()[0] > 0


def test_set_state_clears_a_failed_step():
    t = mps.Tank((18 * L0, 7 * L0, 0.2), (13 * L0, 7 * L0, 6 * L0), L0, 3e-4, row_width=24)
    with pytest.raises(sph.SphError) as e:
        t.step(1)
    assert e.value.code == sph.SPH_ESTATE
    # a state whose rows fit: three of four particles out of the grid, where they stay frozen
    s = t.get_state()
    out = np.arange(t.n) % 4 != 0
    r, u = s["r"].copy(), np.zeros_like(s["u"])
    r[out, 2] = 1e3
    fluid = s["type"] == mps.FLUID
    u[fluid & out] = (0.1, 0.2, 0.3)
    t.set_state(r, u)
    t.step(1)
    s = t.get_state()
    assert np.array_equal(s["u"][fluid & out], u[fluid & out]) and np.array_equal(s["r"][out], r[out])


def test_iteration_cap_is_exact():
    args = ((1.0, 0.5, 0.5), (0.4, 0.5, 0.3), L0, 8e-4)
    its = mps.Tank(*args).pressure()["iterations"]
    assert its > 1
    assert mps.Tank(*args, cg_max=its).pressure()["iterations"] == its
    with pytest.raises(sph.SphError) as e:
        mps.Tank(*args, cg_max=its - 1).pressure()
    assert e.value.code == sph.SPH_EUNSTABLE
