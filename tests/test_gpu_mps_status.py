"""Failed MPS steps (the bounded waits of the CG solve, its iteration cap, the handle
after a failure once a state is loaded) and which neighbour passes a step takes."""
import numpy as np
import pytest
import torch

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


def _lists_overflowed(t):
    """Word 5 of the handle's counters in its workspace (in-grid particles, non-empty
    cells, status, two zeros, the flag, zeros; on a 256-byte boundary)."""
    rows = t.workspace[: t.workspace.numel() // 256 * 256].view(torch.int32).view(-1, 64)
    hit = (rows[:, 0] == t.n) & (rows[:, 1] > 0) & (rows[:, 2] == 0) & (rows[:, 6:16] == 0).all(1)
    hit &= (rows[:, 5] == 0) | (rows[:, 5] == 1)
    at = torch.nonzero(hit).flatten()
    assert len(at) == 1
    return int(rows[at[0], 5])


@pytest.mark.parametrize("width,over", [(64, 0), (32, 0), (31, 1)])
def test_which_neighbour_passes_run(width, over):
    # the shallow pool of test_gpu_mps_rows.py: a floor particle has 32 particles within
    # r_e, so that 31 entries leave the passes to the kernels that search by themselves
    t = mps.Tank((18 * L0, 7 * L0, 0.2), (13 * L0, 7 * L0, 2 * L0), L0, 3e-4, row_width=width)
    t.pressure()
    assert _lists_overflowed(t) == over
