"""The fixed-point factor of the Bulirsch-Stoer pulls over the changeover zone and at its ends: pairs at
separations from far inside to just outside their critical radius (K = 0 up to 0.1 rc, 1 from rc on),
with radii that put the zone's inner boundary on every power-of-two alignment, heavy and massless
partners, a body within rc of the central mass, and kmode 1 (the FP64 form). The pulls are strong (10^-3 solar masses) and
the interval short, so that an error of 1e-8 in a factor would show.

Bound: the BS accepts a component when two extrapolations agree to 1e-12 of |x| or |v|; twice that,
for the rounding of the two sides' sums.
"""
import numpy as np
import pytest

import oracle as O
from paper_1404_2324_gb300 import genga, ics
from tests.gpu_util import aos, dev, soa
from tests.test_gpu_phases import _clumps

pytestmark = pytest.mark.gpu

FRACTIONS = [0.05, 0.0999999, 0.1, 0.1000001, 0.11, 0.2, 0.55, 0.9, 0.999999, 1.0, 1.000001, 1.3]


def _pairs(size, rc_lo, rc_hi, seed, mass):
    rng = np.random.default_rng(seed)
    xs, vs, ms, rcs, groups = [], [], [], [], []
    for k, f in enumerate(FRACTIONS):
        rc = np.exp(rng.uniform(np.log(rc_lo), np.log(rc_hi)))
        a = 0.5 + 0.2 * k
        ang = 2.0 * k
        c = a * np.array([np.cos(ang), np.sin(ang), 0.01])
        vc = np.sqrt(ics.G_GAUSS / a) * np.array([-np.sin(ang), np.cos(ang), 0.0])
        groups.append(np.arange(len(ms), len(ms) + size, dtype=np.int32))
        for q in range(size):
            d = rng.normal(size=3)
            xs.append(c + (0 if q == 0 else f * rc) * d / np.linalg.norm(d))
            vs.append(vc * (1 + 1e-3 * q))
            ms.append(mass if q != 1 else mass * 1e-3)
            rcs.append(rc * (1.0 if q == 0 else 0.7))
    return np.array(xs), np.array(vs), np.array(ms), np.array(rcs), groups


@pytest.mark.parametrize("kmode", [0, 1])
@pytest.mark.parametrize("size,mass,rc", [(2, 1e-3, (0.01, 0.08)), (2, 0.0, (0.01, 0.08)), (3, 1e-3, (0.02, 0.3)), (2, 1e-3, (0.6, 2.4)),
                                          (6, 1e-4, (0.02, 0.3)), (12, 1e-4, (0.02, 0.3)), (40, 1e-5, (0.02, 0.3))])
def test_pulls_across_the_changeover_zone_match_the_oracle(kmode, size, mass, rc):
    x, v, m, r, groups = _pairs(size, *rc, seed=size, mass=mass)
    n, tau = len(m), 0.002
    R, alive = np.zeros(n), np.ones(n, np.int32)
    p = O.params(G=ics.G_GAUSS, m0=1.0, kmode=kmode)
    rx, rv = x.copy(), v.copy()
    for g in groups:
        out = O.bs_group(p, g, tau, m, R, alive, rx, rv, r)
        assert out["status"] == 0
        rx, rv = out["x"], out["v"]
    start = np.concatenate([[0], np.cumsum([len(g) for g in groups])]).astype(np.int32)
    X, V, M, RR, AL = soa(x), soa(v), dev(m), dev(R), dev(alive)
    st, U = genga.genga_phase_bs(n, ics.G_GAUSS, 1.0, tau, 1e-12, 8, 30, kmode, 0, len(groups), dev(start),
                                 dev(np.concatenate(groups)), dev(r), M, RR, AL, X, V)
    assert st == 0
    for got, want in ((aos(X), rx), (aos(V), rv)):
        err = np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)
        assert err.max() <= 2e-12, (err.max(), int(err.argmax()))


@pytest.mark.parametrize("seed,spread,R", [(1, 0.0002, None), (8, 0.0002, None), (4, 0.0003, 2e-5), (6, 0.0003, 2e-5)])
def test_groups_of_three_and_four_with_failed_attempts_match_the_oracle(seed, spread, R):
    """Tight groups of three and four members, up to nine substeps with failed attempts between them
    and, with the larger radii, mergers: from the second attempt on the attempt at H/2 runs in the
    other half of the CTA and is taken exactly when the serial control would try it next. A close
    pass amplifies rounding, so the bound per group is the oracle's own sensitivity: ten times the
    largest change of its result under four changes of the start by 1e-16, and 1e-11 at least."""
    x, v, m, Rr, groups = _clumps((3, 4) * 4, seed=seed, spread=spread, R=R)
    n = len(m)
    alive, rc = np.ones(n, np.int32), np.full(n, 0.02)
    p = O.params(G=ics.G_GAUSS, m0=1.0)
    steps = coll = 0
    for g in groups:
        g = np.asarray(g, np.int32)
        want = O.bs_group(p, g, 6.0, m, Rr, alive, x, v, rc)
        live = g[want["alive"][g] == 1]
        sens = 0.0
        for k in range(4):
            x2 = x * (1 + 1.1e-16 * np.random.default_rng(k).integers(-1, 2, x.shape))
            o = O.bs_group(p, g, 6.0, m, Rr, alive, x2, v, rc)
            sens = max(sens, np.abs(o["x"] - want["x"])[live].max(), np.abs(o["v"] - want["v"])[live].max() / 0.017)
        X, V, M, RR, AL = soa(x), soa(v), dev(m), dev(Rr), dev(alive)
        st, U = genga.genga_phase_bs(n, ics.G_GAUSS, 1.0, 6.0, 1e-12, 8, 30, 0, 1, 1, dev(np.array([0, len(g)], np.int32)),
                                     dev(g), dev(rc), M, RR, AL, X, V)
        assert st == 0
        np.testing.assert_array_equal(AL.cpu().numpy()[g], want["alive"][g])
        err = max(np.abs(aos(X) - want["x"])[live].max(), np.abs(aos(V) - want["v"])[live].max() / 0.017)
        assert err <= max(1e-11, 10 * sens), (err, sens)
        steps += want["bs_steps"]
        coll += len(want["collisions"])
    assert steps > len(groups) and (coll > 0) == (R is not None)


@pytest.mark.parametrize("seed", [4, 6, 9, 13])
def test_mergers_of_groups_of_three_and_four_book_energy_mass_and_radius(seed):
    """The inputs above whose members merge: per group the same mergers as the oracle, the survivors'
    masses and radii, and the internal energy to ten times the oracle's own sensitivity (1e-9 at least,
    the bound of the other groups' mergers)."""
    x, v, m, Rr, groups = _clumps((3, 4) * 4, seed=seed, spread=0.0003, R=2e-5)
    n = len(m)
    alive, rc = np.ones(n, np.int32), np.full(n, 0.02)
    p = O.params(G=ics.G_GAUSS, m0=1.0)
    coll = 0
    for g in groups:
        g = np.asarray(g, np.int32)
        want = O.bs_group(p, g, 6.0, m, Rr, alive, x, v, rc)
        if not len(want["collisions"]):
            continue
        sens = 0.0
        for k in range(4):
            x2 = x * (1 + 1.1e-16 * np.random.default_rng(k).integers(-1, 2, x.shape))
            sens = max(sens, abs(O.bs_group(p, g, 6.0, m, Rr, alive, x2, v, rc)["U"] - want["U"]))
        X, V, M, RR, AL = soa(x), soa(v), dev(m), dev(Rr), dev(alive)
        st, U = genga.genga_phase_bs(n, ics.G_GAUSS, 1.0, 6.0, 1e-12, 8, 30, 0, 1, 1, dev(np.array([0, len(g)], np.int32)),
                                     dev(g), dev(rc), M, RR, AL, X, V)
        assert st == 0
        np.testing.assert_array_equal(AL.cpu().numpy(), want["alive"])
        np.testing.assert_allclose(M.cpu().numpy(), want["m"], rtol=1e-15)
        np.testing.assert_allclose(RR.cpu().numpy(), want["R"], rtol=1e-14)
        assert abs(U - want["U"]) <= max(1e-9 * abs(want["U"]), 10 * sens), (U, want["U"], sens)
        coll += len(want["collisions"])
    assert coll > 0
