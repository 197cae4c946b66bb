"""The Kepler solve where its shortened form hands over or runs out of range: units in which the universal
variable is tiny, and callers that allow few iterations."""
import numpy as np
import pytest
import torch

from paper_1404_2324_gb300 import genga, ics
from tests.gpu_util import aos, dev, soa

pytestmark = pytest.mark.gpu
G = ics.G_GAUSS


def _orbits(n, e_max, seed=7):
    """Orbits of 0.3-5 AU at random phases: x, v, periods."""
    rng = np.random.default_rng(seed)
    a, e = np.exp(rng.uniform(np.log(0.3), np.log(5.0), n)), rng.uniform(0, e_max, n)
    E, w, inc = rng.uniform(0, 2 * np.pi, (3, n))
    inc = 0.2 * inc / (2 * np.pi)
    b, nu = np.sqrt(1 - e * e), np.sqrt(G / a ** 3) / (1 - e * np.cos(E))
    p, q, u, s = a * (np.cos(E) - e), a * b * np.sin(E), -a * np.sin(E) * nu, a * b * np.cos(E) * nu
    turn = lambda p, q: np.stack([p * np.cos(w) - q * np.sin(w), (p * np.sin(w) + q * np.cos(w)) * np.cos(inc),  # noqa: E731
                                  (p * np.sin(w) + q * np.cos(w)) * np.sin(inc)], 1)
    return turn(p, q), turn(u, s), 2 * np.pi * np.sqrt(a ** 3 / G)


def _drift(mu, dt, maxit, x, v):
    n = len(x)
    X, V, fail = soa(x), soa(v), dev(np.zeros(n, np.int32))
    genga.genga_phase_kepler(n, mu, dt, maxit, dev(np.ones(n, np.int32)), X, V, fail)
    torch.cuda.synchronize()
    return aos(X), aos(V), fail.cpu().numpy()


@pytest.mark.parametrize("p", [10, 30, 38, 42, -30])
@pytest.mark.parametrize("dt", [6.0, -20.0])
def test_drift_is_the_same_in_other_units_of_length(p, dt):
    """Lengths 2^p times as large in number (p = 42: AU to 0.03 m; the universal variable goes to 10^-13):
    every operation scales by a power of two, so the results are the same to the last bit."""
    x, v, _ = _orbits(20000, 0.3)
    x0, v0, f0 = _drift(G, dt, 30, x, v)
    x1, v1, f1 = _drift(np.ldexp(G, 3 * p), dt, 30, np.ldexp(x, p), np.ldexp(v, p))
    assert not f0.any() and not f1.any()
    np.testing.assert_array_equal(np.ldexp(x1, -p), x0)
    np.testing.assert_array_equal(np.ldexp(v1, -p), v0)


def _stumpff(z):
    k = np.maximum(0, np.ceil(np.log(np.maximum(np.abs(z), 1e-300) / 0.1) / np.log(4.0))).astype(int)
    z = z / 4.0 ** k
    c2, c3, t2, t3 = 0 * z, 0 * z, 0.5 + 0 * z, 1 / 6 + 0 * z
    for m in range(1, 10):
        c2, c3 = c2 + t2, c3 + t3
        t2, t3 = -t2 * z / ((2 * m + 1) * (2 * m + 2)), -t3 * z / ((2 * m + 2) * (2 * m + 3))
    c1, c0 = 1 - z * c3, 1 - z * c2
    for r in range(k.max()):
        on = k > r
        c0, c1, c2, c3 = (np.where(on, n, o) for n, o in ((2 * c0 * c0 - 1, c0), (c0 * c1, c1), (c1 * c1 / 2, c2), ((c2 + c0 * c3) / 4, c3)))
    return c0, c1, c2, c3


def _converges(x, v, dt, maxit):
    """The plain iteration: single-precision root, one Halley step, Newton steps to 4 ulp."""
    r0, u = np.linalg.norm(x, axis=1), (x * v).sum(1)
    beta = 2 * G / r0 - (v * v).sum(1)
    with np.errstate(all="ignore"):
        s, ok = np.float32(dt / r0), np.zeros(len(x), bool)
        fr, fu, fb, fm, fd = (np.float32(q) for q in (r0, u, beta, G, dt))
        for _ in range(12):
            c0, c1, c2, c3 = (np.float32(c) for c in _stumpff(np.float64(fb * s * s)))
            ds = (fr * s * c1 + fu * s * s * c2 + fm * s * s * s * c3 - fd) / (fr * c0 + fu * s * c1 + fm * s * s * c2)
            s = np.where(ok, s, s - ds)
            ok |= np.abs(ds) <= np.float32(2e-6) * np.abs(s)
        s, done, last = np.where(ok, np.float64(s), dt / r0), np.zeros(len(x), bool), np.full(len(x), 3e38)
        for it in range(maxit):
            c0, c1, c2, c3 = _stumpff(beta * s * s)
            F, Fp = r0 * s * c1 + u * s * s * c2 + G * s ** 3 * c3 - dt, r0 * c0 + u * s * c1 + G * s * s * c2
            ds = F / Fp
            if it == 0:
                ds = np.where(ok, 2 * F * Fp / (2 * Fp * Fp - F * ((G - beta * r0) * s * c1 + u * c0)), ds)
            s = np.where(done, s, s - ds)
            done |= (np.abs(ds) <= 8.9e-16 * np.abs(s)) | ((np.abs(ds) <= 1e-10 * np.abs(s)) & (np.abs(ds) >= 0.5 * last))
            last = np.abs(ds)
    return done


@pytest.mark.parametrize("maxit", [3, 4, 30])
def test_few_iterations_solve_what_the_plain_iteration_solves(maxit):
    """Orbits up to e = 0.99 over up to two periods with a cap on the iterations: no more solves fail than
    of the plain iteration (a tenth and ten more for the rounding of the two)."""
    x, v, P = _orbits(20000, 0.99)
    order = np.argsort(P)
    failed = plain = 0
    for block in np.array_split(order, 50):  # one dt a call: blocks of like periods, 0.01-2 of them
        dt = P[block].mean() * 10.0 ** np.random.default_rng(int(block[0])).uniform(-2, 0.3)
        failed += int(_drift(G, dt, maxit, x[block], v[block])[2].sum())
        plain += int((~_converges(x[block], v[block], dt, maxit)).sum())
    print(f"maxit {maxit}: {failed} failed, of the plain iteration {plain}")
    assert failed <= 1.1 * plain + 10
