"""The fixed-point kick of systems whose radii span many octaves: a few bodies far outside the others are
left out of the grid and their pairs taken in FP64, so that they neither spoil the accuracy of the rest
nor turn every pair into a near one. Bound and oracle as in test_gpu_kick_fixed.py, whose other inputs
run here at the sizes of two to seven tiles, too (its n = 40 is the FP64 kernel's)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1404_2324_gb300 import genga, ics
from paper_1404_2324_gb300.adjoint import AdjointEngine
from tests.gpu_util import pair_sims, rel_state_error, with_central
from tests.test_gpu_kick_fixed import _case, _disk, _run

pytestmark = pytest.mark.gpu


def _spread(kind, n):
    G, m, x, v = _disk(n)
    rng = np.random.default_rng(n)
    if kind.startswith("far"):          # this many at 1000-9000 AU
        k = rng.choice(n, min(int(kind[3:]), n - 2), replace=False)
        d = rng.normal(size=(len(k), 3))
        x[k] = d / np.linalg.norm(d, axis=1)[:, None] * rng.uniform(1e3, 9e3, len(k))[:, None]
    elif kind.startswith("share"):      # this percentage at log-uniform radii 4-40000 AU
        k = rng.choice(n, n * int(kind[5:]) // 100, replace=False)
        x[k] *= np.exp(rng.uniform(0.0, np.log(1e4), len(k)))[:, None]
    elif kind == "octaves":             # one body an octave outwards, to 2^30 times the disk
        k = np.arange(0, n, max(1, n // 30))[:30]
        x[k] *= (2.0 ** np.arange(len(k)))[:, None]
    elif kind == "mixed":               # half of them spread, with ghosts, massless bodies and masses over decades
        k = rng.choice(n, n // 2, replace=False)
        x[k] *= np.exp(rng.uniform(0.0, np.log(1e4), len(k)))[:, None]
        m *= 10.0 ** rng.uniform(-12, 0, n)
        m[1::5] = 0.0
    elif kind == "inner":               # one body an octave inwards, to the central mass
        k = np.arange(0, n, max(1, n // 30))[:30]
        x[k] *= (0.5 ** np.arange(len(k)))[:, None]
        x[-1] = 0.0
    alive = np.ones(n, np.int32)
    if kind == "mixed":
        alive[::4] = 0
    return G, m, alive, x, np.full(n, 0.02)


def _check(G, m, alive, x, rc, kmode=0):
    n = len(m)
    p = O.params(G=G, m0=1.0, dt=6.0, kmode=kmode)
    a, cand = _run(G, m, alive, x, rc, kmode=kmode)
    live = alive == 1
    want = O.accel_B(p, m, alive, x, rc)
    np.testing.assert_array_equal(cand, np.asarray(O.precheck(p, alive, x, rc)).reshape(-1, 2))
    r = np.linalg.norm(x[None] - x[:, None], axis=-1)
    np.fill_diagonal(r, np.inf)
    bound = 2.0 ** -53 * (1.2 * n + 60) * (G * np.where(live, m, 0.0)[None] / r ** 2).sum(1)
    err = np.linalg.norm(a - want, axis=1)
    assert np.all(err[live] <= bound[live]), np.max(err[live] / bound[live])


@pytest.mark.parametrize("n", [70, 97, 200, 257, 1100, 2048])
@pytest.mark.parametrize("kind", ["far1", "far3", "far40", "share10", "share50", "share100", "octaves", "inner", "mixed"])
def test_kick_of_radii_over_many_octaves(kind, n):
    _check(*_spread(kind, n))


@pytest.mark.parametrize("n", [70, 97, 200])
@pytest.mark.parametrize("kind", ["decades", "giant", "outlier", "ghosts", "massless"])
def test_kick_of_a_few_tiles(kind, n):
    _check(*_case(kind, n))


@pytest.mark.parametrize("n", [100, 300])
def test_steps_of_a_scattered_disk_match_the_oracle(n):
    """A third of the bodies out to 4000 AU on the orbits of their new distance: one step of the main mode
    (its opening kick weighs every pair) and of the differentiable engine."""
    d = ics.disk2048(9, n=n, total_mass=2 * ics.M_EARTH * n / 2048)
    rng = np.random.default_rng(n)
    k = rng.choice(n, n // 3, replace=False)
    f = np.exp(rng.uniform(0.0, np.log(1e3), len(k)))[:, None]
    d["x"][k] *= f
    d["v"][k] /= np.sqrt(f)
    g, o = pair_sims(d, 4, steps=1)
    err, same = rel_state_error(g, o)
    g.close()
    o.close()
    assert same and err <= 1e-12
    o = O.Sim(O.params(G=d["G"], m0=1.0, dt=d["dt"], order=2, collisions=0), d["m"], np.zeros(n), d["x"], d["v"])
    o.step(1)
    want = o.state()
    o.close()
    eng = AdjointEngine(np.ones(1), d["G"], d["dt"], 2, ckpt_every=1)
    t = lambda q: torch.tensor(q[None], dtype=torch.float64, device="cuda")  # noqa: E731
    xo, vo = eng.forward(t(d["x"]), t(d["v"]), t(d["m"]), 1)
    eng.close()
    for got, ref in ((xo, want["x"]), (vo, want["v"])):
        assert np.max(np.linalg.norm(got[0].cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)) <= 1e-12


def _kick_us(x, d):
    m, R, x0, v = with_central({**d, "x": x})
    h = genga.genga_init(m, R, x0, v, d["G"], 6.0, 2)
    genga.genga_set_profiling(h, True)
    t = []
    for _ in range(20):
        genga.genga_step(h, 1)
        ms, launches = genga.genga_kick_time(h)
        t.append(ms / launches * 1e3)
    genga.genga_free(h)
    return min(t)


def test_a_far_body_does_not_slow_the_kick():
    """2048 bodies with one and with eight of them at 3000 AU, against the same disk: with every pair of
    their CTAs in FP64 the kick took more than four times as long; twice is the bound."""
    d = ics.disk2048(3)
    plain = _kick_us(d["x"], d)
    for k in (1, 8):
        x = d["x"].copy()
        x[:: 2048 // k] *= 3000.0 / np.linalg.norm(x[:: 2048 // k], axis=1)[:, None]
        assert _kick_us(x, d) <= 2.0 * plain
