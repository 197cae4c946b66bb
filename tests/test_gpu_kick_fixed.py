"""The fixed-point pair kernel (the default kick) against the oracle's direct sum, at the sizes and
inputs where it changes its shape or its path: one tile to many, chunks of every length, bodies the
grid does not resolve (pairs much closer than the system is wide), masses over many decades, ghosts,
massless bodies, and numbers the fixed-point form cannot hold.

Bound per body, fixed beforehand: a term carries at most 6 roundings (position difference, r^2,
r^-3, product) and the sums of n terms at most n/8 + 32 more on the way (chunk sums, the sum over
chunks), each 2^-53 of the sum of the terms' magnitudes; the oracle's own plain sum adds n + 6.
"""
import numpy as np
import pytest

import oracle as O
from paper_1404_2324_gb300 import genga, ics
from tests.gpu_util import aos, dev, soa

pytestmark = pytest.mark.gpu


def _disk(n, seed=5):
    d = ics.disk2048(seed, n=max(n, 4), total_mass=2 * ics.M_EARTH * n / 2048)
    return d["G"], d["m"][:n].copy(), d["x"][:n].copy(), d["v"][:n].copy()


def _case(kind, n):
    G, m, x, v = _disk(n)
    rng = np.random.default_rng(n)
    alive = np.ones(n, np.int32)
    if kind == "decades":
        m *= 10.0 ** rng.uniform(-25, 0, n)
    elif kind == "giant":
        m[n // 2] = 1e-3
    elif kind == "outlier":      # the grid of the whole no longer resolves the close pairs
        x[0] *= 1e4
        for k in range(1, n - 1, 7):
            x[k + 1] = x[k] * (1 + 1e-7)
    elif kind == "ghosts":
        alive[::3] = 0
    elif kind == "massless":
        m[1::2] = 0.0
    p = O.params(G=G, m0=1.0, dt=6.0)
    rc = O.rcrit(p, 6.0, m, alive, x, v)
    if kind == "outlier":
        rc *= 1e-6               # far pairs down to 1e-7 AU
    return G, m, alive, x, rc


def _run(G, m, alive, x, rc, precise=0, kmode=0):
    n = len(m)
    cap = max(1, n * (n - 1) // 2)
    a, cand = dev(np.zeros((3, n))), dev(np.zeros(2 * cap, np.int32))
    cnt = genga.genga_phase_kick(n, G, 3.0, kmode, precise, dev(m), dev(alive), soa(x), dev(rc), a, cand, cap)
    return aos(a), cand.cpu().numpy()[: 2 * cnt].reshape(-1, 2)


@pytest.mark.parametrize("kind,n", [("disk", n) for n in (1, 2, 31, 32, 33, 64, 65, 129, 224, 225, 256, 257, 511, 1000, 2017, 2048)]
                         + [(k, n) for k in ("decades", "giant", "outlier", "ghosts", "massless") for n in (40, 300, 1100)])
def test_fixed_point_kick_matches_the_direct_sum(kind, n):
    G, m, alive, x, rc = _case(kind, n)
    p = O.params(G=G, m0=1.0, dt=6.0)
    a, cand = _run(G, m, alive, x, rc)
    live = alive == 1
    want = O.accel_B(p, m, alive, x, rc)
    np.testing.assert_array_equal(cand, np.asarray(O.precheck(p, alive, x, rc)).reshape(-1, 2))
    r = np.linalg.norm(x[None] - x[:, None], axis=-1)
    np.fill_diagonal(r, np.inf)
    t = G * np.where(live, m, 0.0)[None] / r ** 2
    bound = 2.0 ** -53 * (1.2 * n + 60) * t.sum(1)
    err = np.linalg.norm(a - want, axis=1)
    assert np.all(err[live] <= bound[live]), (kind, n, np.max(err[live] / bound[live]))


def test_fixed_point_kick_passes_on_numbers_it_cannot_hold():
    """A position or mass that is not finite reaches the bodies it touches as in the FP64 kernel, and
    a negative mass pushes."""
    G, m, alive, x, rc = _case("disk", 70)
    for what in ("nan", "inf mass", "negative"):
        m2, x2 = m.copy(), x.copy()
        if what == "nan":
            x2[5, 1] = np.nan
        elif what == "inf mass":
            m2[5] = np.inf
        else:
            m2[5] = -m2[5]
        a, _ = _run(G, m2, alive, x2, rc)
        b, _ = _run(G, m2, alive, x2, rc, precise=1)
        np.testing.assert_array_equal(np.isfinite(a), np.isfinite(b), err_msg=what)
        f = np.isfinite(a) & np.isfinite(b)
        np.testing.assert_allclose(a[f], b[f], rtol=0, atol=1e-13 * np.abs(b[f]).max() if f.any() else 0, err_msg=what)


@pytest.mark.parametrize("precise", [0, 1])
def test_kick_without_allocation_clears_its_scratch_between_sizes(precise):
    """Calls of rising and falling size, one after the other on the one scratch array: each gives the
    allocating kick's numbers and candidates, so nothing of the call before is left."""
    import torch

    for n in (1024, 1, 33, 1000, 31, 32, 65, 1023, 2):
        G, m, alive, x, rc = _case("ghosts" if n % 2 else "disk", n)
        cap = max(1, n * (n - 1) // 2)
        want, pairs = _run(G, m, alive, x, rc, precise)
        a, cand, cnt = dev(np.zeros((3, n))), dev(np.zeros(2 * cap, np.int32)), dev(np.zeros(1, np.int32))
        genga.genga_kick_noalloc(n, G, 3.0, 0, precise, dev(m), dev(alive), soa(x), dev(rc), a, cand, cap, cnt)
        torch.cuda.synchronize()
        assert int(cnt.item()) == len(pairs), n
        np.testing.assert_array_equal(cand.cpu().numpy()[: 2 * len(pairs)].reshape(-1, 2), pairs, err_msg=str(n))
        live = alive == 1
        np.testing.assert_array_equal(aos(a)[live], want[live], err_msg=str(n))


@pytest.mark.parametrize("n", [40, 300, 1025])
@pytest.mark.parametrize("precise", [0, 1])
def test_rows_of_many_near_partners_are_summed_in_full(n, precise):
    """Critical radii so wide that a body has far more than 32 near partners, on both sides of the
    changeover. A near term carries about 20 roundings, counted in the bound's constant."""
    G, m, alive, x, rc = _case("ghosts", n)
    rc = np.where(alive == 1, 0.6, 0.0)
    p = O.params(G=G, m0=1.0, dt=6.0)
    a, cand = _run(G, m, alive, x, rc, precise)
    want = O.accel_B(p, m, alive, x, rc)
    np.testing.assert_array_equal(cand, np.asarray(O.precheck(p, alive, x, rc)).reshape(-1, 2))
    live = alive == 1
    r = np.linalg.norm(x[None] - x[:, None], axis=-1)
    np.fill_diagonal(r, np.inf)
    t = G * np.where(live, m, 0.0)[None] / r ** 2
    assert n < 300 or np.bincount(cand.ravel()).max() > 40
    err = np.linalg.norm(a - want, axis=1)
    assert np.all(err[live] <= (2.0 ** -53 * (1.2 * n + 100) * t.sum(1))[live]), np.max(err / t.sum(1))
