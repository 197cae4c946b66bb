"""Bodies at one position with one velocity. Their mutual pull is a factor times a separation of zero, so
they go on together as each would alone (or merge): the Bulirsch-Stoer kernels of every group size,
the batched schedules and the differentiable engine. The other members lie outside each other's
critical radii, so that no sum rounds differently for the two.

Bound: the BS accepts a component when two extrapolations agree to 1e-12 of |x| or |v|; twice that.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1404_2324_gb300 import genga, ics
from paper_1404_2324_gb300.adjoint import AdjointEngine
from tests.gpu_util import aos, dev, soa

pytestmark = pytest.mark.gpu
G = ics.G_GAUSS


def _spaced(n, mass=3e-7):
    """n bodies on circular orbits, rings of 20 apart by more than 0.2 AU; 0 and 1 at one place."""
    k = np.maximum(np.arange(n) - 1, 0)
    a, ang = 1.0 + 0.5 * (k // 20), 2 * np.pi * (k % 20) / 20
    x = a[:, None] * np.stack([np.cos(ang), np.sin(ang), 0 * ang], 1)
    v = np.sqrt(G / a)[:, None] * np.stack([-np.sin(ang), np.cos(ang), 0 * ang], 1)
    return x, v, np.full(n, mass)


def _close(got, want):
    return np.max(np.linalg.norm(got - want, axis=-1) / np.linalg.norm(want, axis=-1)) <= 2e-12


def _phase(x, v, m, R, collisions):
    n = len(m)
    X, V, M, AL = soa(x), soa(v), dev(m), dev(np.ones(n, np.int32))
    st, _ = genga.genga_phase_bs(n, G, 1.0, 6.0, 1e-12, 8, 30, 0, collisions, 1, dev(np.array([0, n], np.int32)),
                                 dev(np.arange(n, dtype=np.int32)), dev(np.full(n, 0.02)), M, dev(R), AL, X, V)
    assert st == 0, st
    return aos(X), aos(V), M.cpu().numpy(), AL.cpu().numpy()


@pytest.mark.parametrize("n", [2, 3, 4, 5, 12, 30, 40, 150])
def test_coincident_members_go_on_together(n):
    x, v, m = _spaced(n)
    gx, gv, _, _ = _phase(x, v, m, np.zeros(n), 0)
    p = O.params(G=G, m0=1.0)
    for i in range(n):
        out = O.bs_group(p, [i], 6.0, m, np.zeros(n), np.ones(n, np.int32), x, v, np.full(n, 0.02))
        assert _close(gx[i], out["x"][i]) and _close(gv[i], out["v"][i]), i
    np.testing.assert_array_equal(gx[0], gx[1])
    np.testing.assert_array_equal(gv[0], gv[1])


@pytest.mark.parametrize("n", [2, 3, 6, 40])
def test_coincident_members_merge_on_contact(n):
    x, v, m = _spaced(n)
    R = np.zeros(n)
    R[:2] = 1e-5
    gx, gv, gm, al = _phase(x, v, m, R, 1)
    assert al[:2].sum() == 1 and al[2:].all()
    k = int(np.argmax(al[:2]))
    assert gm[k] == 2 * m[0]
    out = O.bs_group(O.params(G=G, m0=1.0), [0], 6.0, m, np.zeros(n), np.ones(n, np.int32), x, v, np.full(n, 0.02))
    assert _close(gx[k], out["x"][0]) and _close(gv[k], out["v"][0])


def _one_heavier(m, x, v, steps):
    """The oracle's run of one body of twice the mass (the pair's common motion)."""
    s = O.Sim(O.params(G=G, m0=1.0, dt=6.0, order=2, collisions=0), 2 * m[:1], np.zeros(1), x[:1], v[:1])
    s.step(steps)
    st = s.state()
    s.close()
    return st["x"][0], st["v"][0]


@pytest.mark.parametrize("persistent", [0, 1])
def test_coincident_pair_in_a_batch(persistent):
    x, v, m = _spaced(2)
    xx, vv, mm = np.concatenate([x, 1.1 * x]), np.concatenate([v, v]), np.concatenate([m, m])
    h = genga.genga_init_batch(np.array([0, 2, 4]), np.ones(2), mm, np.zeros(4), xx, vv, G, 6.0, 2, 1)
    try:
        genga.genga_batch_set_schedule(h, persistent)
        genga.genga_set_state_batch(h, xx, vv)
        genga.genga_step(h, 2)
        g = genga.genga_get_state_batch(h, 4)
        assert genga.genga_status(h)[0] & genga.ST_BS_FAILED == 0
        for s in (0, 2):
            wx, wv = _one_heavier(mm[s:], xx[s:], vv[s:], 2)
            for i in (s, s + 1):
                assert _close(g["x"][i], wx) and _close(g["v"][i], wv), i
    finally:
        genga.genga_free(h)


def test_coincident_pair_in_the_differentiable_engine():
    x, v, m = _spaced(2)
    t = lambda q: torch.tensor(q[None], dtype=torch.float64, device="cuda")  # noqa: E731
    eng = AdjointEngine(np.ones(1), G, 6.0, 2, ckpt_every=1)
    xo, vo = eng.forward(t(x), t(v), t(m), 2)
    assert eng.status() & 0x2A == 0
    wx, wv = _one_heavier(m, x, v, 2)
    gx, gv, _ = eng.backward(torch.ones_like(xo), torch.ones_like(vo))
    eng.close()
    for i in (0, 1):
        assert _close(xo[0, i].cpu().numpy(), wx) and _close(vo[0, i].cpu().numpy(), wv)
    assert torch.isfinite(gx).all() and torch.isfinite(gv).all()
