"""Kicks of bodies whose G m lies one unit below a power of two, with separations whose squares lie around
an odd power of two: the ends of the ranges of the fixed-point pull, where a carry loses a term whole.
The main kick and the forward kick of the differentiable engine against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1404_2324_gb300 import genga
from paper_1404_2324_gb300.adjoint import AdjointEngine
from tests.gpu_util import aos, dev, soa

pytestmark = pytest.mark.gpu
G = 2.0 ** -11


def _sphere(n, center, mass, width, p=-1, seed=4):
    """A body at center and n - 1 others at r^2 = 2^p (1 + 2 width u), u in [-1, 1]: m, x."""
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(n, 3))
    d *= (np.sqrt(2.0 ** p) * (1 + width * rng.uniform(-1, 1, n)) / np.linalg.norm(d, axis=1))[:, None]
    d[0] = 0.0
    return np.full(n, mass), np.asarray(center) + d


@pytest.mark.parametrize("n", [65, 200, 1000])
@pytest.mark.parametrize("mantissa", [1 - 2.0 ** -53, 1 - 1e-8, 1 - 1e-7])
def test_kick_at_the_top_of_a_binade(n, mantissa):
    """Bound as in test_gpu_kick_fixed.py."""
    for width in (3e-8, 3e-7):
        m, x = _sphere(n, (0.3, -0.2, 0.1), 2.0 ** -22 * mantissa, width)
        alive, rc = np.ones(n, np.int32), np.full(n, 1e-6)
        p = O.params(G=G, m0=1.0, dt=6.0)
        cap = n
        a, cand = dev(np.zeros((3, n))), dev(np.zeros(2 * cap, np.int32))
        genga.genga_phase_kick(n, G, 3.0, 0, 0, dev(m), dev(alive), soa(x), dev(rc), a, cand, cap)
        want = O.accel_B(p, m, alive, x, rc)
        r = np.linalg.norm(x[None] - x[:, None], axis=-1)
        np.fill_diagonal(r, np.inf)
        bound = 2.0 ** -53 * (1.2 * n + 60) * (G * m[None] / r ** 2).sum(1)
        err = np.linalg.norm(aos(a) - want, axis=1)
        assert np.all(err <= bound), (width, np.max(err / bound))


def test_forward_kick_of_the_differentiable_engine_at_the_top_of_a_binade():
    """The opening kick sees the given positions; one step to 1e-12 (a lost pull is 1e-7 of a velocity)."""
    n = 100
    m, x = _sphere(n, (3.0, 0.0, 0.0), 2.0 ** -20 * (1 - 2.0 ** -53), 3e-8)
    r = np.linalg.norm(x, axis=1)
    v = np.cross([0.0, 0.0, 1.0], x)
    v *= (np.sqrt(G / r) / np.linalg.norm(v, axis=1))[:, None]
    eng = AdjointEngine(np.ones(1), G, 6.0, 2, ckpt_every=1)
    t = lambda q: torch.tensor(q[None], dtype=torch.float64, device="cuda")  # noqa: E731
    xo, vo = eng.forward(t(x), t(v), t(m), 1)
    p = O.params(G=G, m0=1.0, dt=6.0, order=2, collisions=0)
    s = O.Sim(p, m, np.zeros(n), x, v)
    s.step(1)
    want = s.state()
    s.close()
    eng.close()
    for got, ref in ((xo, want["x"]), (vo, want["v"])):
        assert np.max(np.linalg.norm(got[0].cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)) <= 1e-12
