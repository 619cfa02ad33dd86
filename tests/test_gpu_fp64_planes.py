"""The FP64 pair pass next to the coordinate planes, where doubles are finest, and far
from them: mu of single pairs against extended precision, and tanks of any length."""
import numpy as np
import pytest

import oracle
from gpu_common import load_state, normwise, oracle_case
from paper_2306_01959_gb300 import sph, workloads as wl

pytestmark = pytest.mark.gpu

TOL = 2e-14  # two roundings of the FP64 sums of a few hundred terms


@pytest.mark.parametrize("symmetric", [0, 1])
def test_mu_of_pairs_at_the_planes(symmetric):
    # pairs of fluid particles near x = y = z = 0, one at rest and one that flies off
    # so fast that their mu is the largest of both; r from 2h / 64 to 2h / 2
    dp = 0.02
    c = wl.Case("planes", (0.6, 0.6, 0.6), (0.5, 0.5, 0.5), None, dp)
    case = oracle_case(c)
    st = oracle.scene(case)
    rng = np.random.Generator(np.random.PCG64(52))
    h2 = 2.0 * c.h
    f = np.flatnonzero(st.type == oracle.FLUID)
    r, u = st.r.copy(), np.zeros_like(st.u)
    sites = [np.roll((0.0, 0.0, z), k) for z in (0.2, 0.4) for k in range(3)] + [(0.0, 0.0, 0.0)]
    ids = []
    for k, at in enumerate(sites):  # at one to three planes; the pairs do not see each other
        i, j = f[2 * k], f[2 * k + 1]
        plane = rng.uniform(0.0, 0.02, 3)
        r[i] = np.where(np.asarray(at) > 0.0, at, plane * h2)
        d = np.abs(rng.normal(size=3))
        r[j] = r[i] + d / np.linalg.norm(d) * h2 * 2.0 ** -(1 + 5 * k / 6)
        u[j] = (r[j] - r[i]) / np.linalg.norm(r[j] - r[i]) * 1e4
        ids += [i, j]
    sim = sph.Simulation(c, precision=sph.FP64, pair_symmetric=symmetric)
    load_state(sim, oracle.State(r, u, st.rho, st.type))
    mu = sim.derivatives()[2]
    L = np.longdouble
    rl, ul = r.astype(L), u.astype(L)
    eta2 = L(0.01) * L(c.h) * L(c.h)
    for a in ids:  # the largest mu of all pairs of a
        d, v = rl - rl[a], ul - ul[a]
        d2 = (d * d).sum(1)
        m = np.where(d2 < L(h2) * L(h2), L(c.h) * (v * d).sum(1) / (d2 + eta2), 0)
        k = int(np.argmax(m))
        # r_ij and the product with it, 1 + 3 roundings, over what the product cancels (u_ij
        # is exact), the reciprocal, three more products, two of eta^2, and the positions' unit
        cond = float(np.abs(v[k] * d[k]).sum() / (v[k] * d[k]).sum())
        err = float(abs(L(mu[a]) / m[k] - 1))
        assert err <= (4.0 * cond + 6.0) * 2.0**-53 + cond * 2.0**-56, (a, k, err, cond)


@pytest.mark.parametrize("kw", [{}, {"delta_mode": sph.DELTA_FULL_SUPPORT}, {"pair_symmetric": 1}])
def test_length_of_the_tank_does_not_matter(kw):
    # the same column in tanks of 20, 500 and 3000 supports: the same bits (the
    # each-pair-once form adds in any order); and pushed to the far end against the oracle
    h = 0.024
    out = []
    for length in (20.0, 500.0, 3000.0):
        c = wl.Case("long", (2 * h * length, 0.08, 0.1), (0.2, 0.08, 0.06), None, 0.02, h=h)
        case = oracle_case(c, **{k: v for k, v in kw.items() if k == "delta_mode"})
        st = oracle.scene(case)
        nf = int((st.type == oracle.FLUID).sum())
        rng = np.random.Generator(np.random.PCG64(7))
        r, u, rho = st.r.copy(), st.u.copy(), st.rho.copy()
        r[:nf] += rng.normal(0.0, 0.003, (nf, 3))
        u[:nf] = rng.normal(0.0, 0.3, (nf, 3))
        rho[:nf] += rng.normal(0.0, 2.0, nf)
        sim = sph.Simulation(c, precision=sph.FP64, **kw)
        load_state(sim, oracle.State(r, u, rho, st.type))
        out.append([g[:nf].copy() for g in sim.derivatives()])
        far = r.copy()
        far[:nf, 0] += round(c.tank[0] / 0.02) * 0.02 - 0.22
        st = oracle.State(far, u, rho, st.type)
        load_state(sim, st)
        got, ref = sim.derivatives(), oracle.derivatives(case, st)
        assert max(normwise(got[k][:nf], ref[k][:nf]) for k in range(3)) <= TOL
        assert np.array_equal(got[3], ref[3])
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert normwise(a, b) <= TOL if kw.get("pair_symmetric") else np.array_equal(a, b)
