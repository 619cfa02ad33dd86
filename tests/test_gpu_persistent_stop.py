"""The persistent launch after a failed check: it ends before the next update."""
import numpy as np
import pytest
import torch

from paper_2306_01959_gb300 import sph, workloads as wl

pytestmark = pytest.mark.gpu

ST_BOUNDS = 8  # device status bit of a failed index check


def _misc(sim):
    """The handle's counters in its workspace: in-domain particles, non-empty cells,
    status, work queue, tiles, and zeros, on a 256-byte boundary."""
    rows = sim.workspace[: sim.workspace.numel() // 256 * 256].view(torch.int32).view(-1, 64)
    hit = (rows[:, 0] == sim.n) & (rows[:, 1] > 0) & (rows[:, 2] == 0) & (rows[:, 4] > 0)
    hit &= (rows[:, 5:16] == 0).all(1)
    at = torch.nonzero(hit).flatten()
    assert len(at) == 1
    return rows[at[0]]


def test_a_failed_check_ends_the_launch():
    c = wl.small_dambreak()
    sim = sph.Simulation(c, precision=sph.MIXED, persistent=1)
    sim.step(0.0, 3)
    sim.sync()
    before = sim.get_state()
    misc = _misc(sim)
    misc[2] = ST_BOUNDS  # as if a check had failed
    sim.step(0.0, 50)
    with pytest.raises(sph.SphError) as e:
        sim.sync()
    assert e.value.code == sph.SPH_ESTATE
    misc[2] = 0  # (a state is not handed out after a failed check)
    after = sim.get_state()
    for k in ("r", "u", "rho"):
        assert np.array_equal(before[k], after[k]), k
    # a loaded state clears it
    sim.restore(before)
    ref = sph.Simulation(c, precision=sph.MIXED, use_graph=0)
    ref.restore(before)
    for s in (sim, ref):
        s.step(0.0, 5)
        s.sync()
    assert np.array_equal(sim.get_state()["r"], ref.get_state()["r"])
