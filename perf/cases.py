"""The work a user of this library has it do, as cases to be timed and compared.

A case is a dict of plain values; ``kind`` says which public entry points it goes through:

* ``kick``   -- genga_kick_noalloc on device arrays: the weighted pair kick and the prechecker of n
                bodies (the call for latency-critical loops; n up to 1024).
* ``kepler`` -- genga_phase_kepler on device arrays: the Kepler drift of n bodies.
* ``disk``   -- one simulation, host arrays in and out: genga_set_state, genga_step, genga_get_state.
* ``tp``     -- planets and test particles: genga_step, genga_get_state_tp.
* ``batch``  -- many small systems: genga_set_state_batch, genga_step, genga_get_state_batch.
* ``adjoint``-- the differentiable engine: hybrid_steps and its gradient.

A simulation's pass holds as few steps as make the outputs comparable to rounding: close encounters
amplify rounding from step to step.
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_1404_2324_gb300 import adjoint, genga

G = 0.01720209895 ** 2      # AU^3 Msun^-1 day^-2
M_EARTH = 3.00349e-6        # Msun
DT = 6.0                    # days
CAP_PER_BODY = 64           # candidate pairs a kick call has room for, per body


def listed():
    return [
        # one kick of a small system inside a caller's loop: launch latency
        {"name": "kick_64", "kind": "kick", "n": 64, "kmode": 0},
        # the same call near its largest size, not a multiple of 32
        {"name": "kick_1000", "kind": "kick", "n": 1000, "kmode": 0},
        # the drift alone of a swarm of bodies
        {"name": "kepler_200003", "kind": "kepler", "n": 200003},
        # the small disk of the energy-conservation runs: a step is a chain of short kernels
        {"name": "disk_32", "kind": "disk", "n": 32, "order": 2, "n2": 0.4, "steps": 10},
        # a planetesimal disk of middle size, 2nd order
        {"name": "disk_500", "kind": "disk", "n": 500, "order": 2, "n2": 0.4, "steps": 10},
        # the largest disk at 4th order: the benchmark workload
        {"name": "disk_2048_o4", "kind": "disk", "n": 2048, "order": 4, "n2": 0.4, "steps": 4},
        # wide critical radii (the n2 sweep): encounter groups of up to hundreds of bodies
        {"name": "disk_1024_wide", "kind": "disk", "n": 1024, "order": 2, "n2": 1.0, "steps": 2},
        # planets with a modest swarm of test particles
        {"name": "tp_100000", "kind": "tp", "n": 100000, "planets": 8, "order": 2, "steps": 4},
        # planets with a large swarm, 4th order
        {"name": "tp_1048576_o4", "kind": "tp", "n": 1048576, "planets": 8, "order": 4, "steps": 2},
        # a few hundred planetary systems of 4 to 64 bodies
        {"name": "batch_300", "kind": "batch", "systems": 300, "order": 2, "steps": 4},
        # thousands of planetary systems
        {"name": "batch_8192", "kind": "batch", "systems": 8192, "order": 2, "steps": 4},
        # gradients through 20 steps of 64 disks
        {"name": "adjoint_64x256", "kind": "adjoint", "systems": 64, "n": 256, "order": 2, "steps": 20, "every": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["kick", "kepler", "disk", "disk", "tp", "batch", "adjoint"])
    order = rng.choice([2, 2, 4, 6])
    substeps = {2: 1, 4: 3, 6: 7}[order]
    if kind == "kick":
        return {"kind": kind, "n": _log_int(rng, 16, 1024), "kmode": rng.choice([0, 0, 1])}
    if kind == "kepler":
        return {"kind": kind, "n": _log_int(rng, 256, 1 << 18)}
    if kind == "disk":
        return {"kind": kind, "n": _log_int(rng, 16, 2048), "order": order, "n2": rng.choice([0.4, 0.4, 0.7]),
                "steps": max(1, rng.randint(1, 8) // substeps)}
    if kind == "tp":
        return {"kind": kind, "n": _log_int(rng, 1 << 12, 1 << 20), "planets": rng.randint(1, 12), "order": order,
                "steps": max(1, 4 // substeps)}
    if kind == "batch":
        return {"kind": kind, "systems": _log_int(rng, 32, 8192), "order": order, "steps": max(1, 4 // substeps)}
    return {"kind": kind, "systems": _log_int(rng, 1, 64), "n": _log_int(rng, 24, 256), "order": order,
            "steps": max(1, rng.randint(4, 12) // substeps), "every": rng.randint(2, 8)}


# ------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 11)
    return g


def _uniform(g, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _rayleigh(g, n, sigma, most):
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    return (sigma * torch.sqrt(-2.0 * torch.log1p(-u))).clamp(max=most)


def _orbits(g, mu, a, e, inc):
    """Heliocentric positions and velocities [n, 3] of orbits with random angles."""
    n = a.numel()
    node, peri, M = (_uniform(g, n, 0.0, 2.0 * math.pi) for _ in range(3))
    E = M + e * torch.sin(M)
    for _ in range(10):
        E = E - (E - e * torch.sin(E) - M) / (1.0 - e * torch.cos(E))
    b = torch.sqrt(1.0 - e * e)
    w = torch.sqrt(mu / a ** 3) / (1.0 - e * torch.cos(E))
    p, q = a * (torch.cos(E) - e), a * b * torch.sin(E)
    u, v = -a * torch.sin(E) * w, a * b * torch.cos(E) * w
    cO, sO, cw, sw, ci, si = (f(t) for t in (node, peri, inc) for f in (torch.cos, torch.sin))
    P = torch.stack([cO * cw - sO * sw * ci, sO * cw + cO * sw * ci, sw * si], -1)
    Q = torch.stack([-cO * sw - sO * cw * ci, -sO * sw + cO * cw * ci, cw * si], -1)
    return p[:, None] * P + q[:, None] * Q, u[:, None] * P + v[:, None] * Q


def _log_masses(g, n, lo, hi):
    return torch.exp(_uniform(g, n, math.log(lo), math.log(hi)))


def _radii(m):
    """Radii [AU] of bodies of 2 g/cm^3."""
    return torch.pow(m * (1.98847e33 / 2.0) * (3.0 / (4.0 * math.pi)), 1.0 / 3.0) / 1.495978707e13


def _disk(g, n):
    """A planetesimal disk: masses log-uniform (2 Earth masses in 2048 bodies), low e and i; 32
    bodies and fewer as in the small disk of 0.5-1.5 AU."""
    m = _log_masses(g, n, 1e-8, 1e-6)
    if n > 32:
        m = m * (2.0 * M_EARTH * n / 2048 / m.sum())
    a = _uniform(g, n, 0.5, 4.0 if n > 32 else 1.5)
    x, v = _orbits(g, G * (1.0 + m), a, _rayleigh(g, n, 0.01, 0.9), _rayleigh(g, n, 0.005, 1.0))
    return m, x, v


def _rcrit(m, x, v, n1=3.0, n2=0.4):
    """Critical radii of the bodies (Eq. rcrit) for a step of DT."""
    r, v2 = x.norm(dim=1), (v * v).sum(1)
    a = 1.0 / (2.0 / r - v2 / G)
    return torch.maximum(n1 * a * torch.pow(m / 3.0, 1.0 / 3.0), n2 * DT * torch.sqrt(v2))


def _pinned(t):
    """A page-locked host copy (a numpy array) of a tensor."""
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h.numpy()


def _pinned_empty(shape, dtype=torch.float64):
    return torch.zeros(shape, dtype=dtype, pin_memory=True).numpy()


def _central(m, x, v):
    """Host arrays with the central mass in row 0."""
    z, one = torch.zeros(1, 3, dtype=x.dtype, device=x.device), torch.ones(1, dtype=m.dtype, device=m.device)
    R = torch.cat([0.0 * one, _radii(m)])
    return [_pinned(t) for t in (torch.cat([one, m]), R, torch.cat([z, x]), torch.cat([z, v]))]


class _Context:
    """A simulation's handle and its page-locked host buffers."""

    def __init__(self, handle, **buffers):
        self.handle = handle
        self.__dict__.update(buffers)

    def __del__(self):
        genga.genga_free(self.handle)


# ------------------------------------------------------------------------------------ prepare, run
def _sizes(case):
    """Bodies per system, star not counted, as in the many-systems shape: 3 to 63 each."""
    return np.random.default_rng(case["systems"]).integers(3, 64, case["systems"])


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind == "kick":
        n = case["n"]
        m, x, v = _disk(g, n)
        rc = _rcrit(m, x, v)
        new = lambda *s, dtype=torch.int32: torch.zeros(*s, dtype=dtype, device="cuda")  # noqa: E731
        return {"case": case, "m": m, "x": x.T.contiguous(), "rc": rc, "alive": torch.ones(n, dtype=torch.int32, device="cuda"),
                "a": new(3, n, dtype=torch.float64), "cand": new(CAP_PER_BODY * n, 2), "ncand": new(1)}
    if kind == "kepler":
        n = case["n"]
        a = _uniform(g, n, 0.3, 5.0)
        x, v = _orbits(g, G, a, _uniform(g, n, 0.0, 0.3), _uniform(g, n, 0.0, 0.2))
        return {"case": case, "x": x.T.contiguous(), "v": v.T.contiguous(), "alive": torch.ones(n, dtype=torch.int32, device="cuda"),
                "fail": torch.zeros(n, dtype=torch.int32, device="cuda")}
    if kind == "disk":
        n = case["n"] + 1
        m, R, x, v = _central(*_disk(g, case["n"]))
        h = genga.genga_init(m, R, x, v, G, DT, case["order"])
        if case["n2"] != 0.4:
            p = genga.genga_default_params()
            p.n2 = case["n2"]
            genga.genga_set_params(h, p)
        out = dict(x=_pinned_empty((n, 3)), v=_pinned_empty((n, 3)), m=_pinned_empty(n), R=_pinned_empty(n),
                   alive=_pinned_empty(n, torch.int32))
        return {"case": case, "ctx": _Context(h, x=x, v=v, out=out)}
    if kind == "tp":
        k, n = case["planets"], case["n"]
        m = _log_masses(g, k, 1e-7, 1e-4)
        a = torch.logspace(math.log10(0.4), math.log10(30.0), k, dtype=torch.float64, device="cuda")
        x, v = _orbits(g, G * (1.0 + m), a, _rayleigh(g, k, 0.01, 0.9), _rayleigh(g, k, 0.01, 1.0))
        xt, vt = _orbits(g, G, _uniform(g, n, 0.3, 5.0), _uniform(g, n, 0.0, 0.3), _uniform(g, n, 0.0, 0.2))
        h = genga.genga_init_tp(*_central(m, x, v), G, DT, case["order"], _pinned(xt), _pinned(vt), np.zeros(n))
        return {"case": case, "ctx": _Context(h, xt=_pinned_empty((n, 3)), vt=_pinned_empty((n, 3)),
                                              alive=_pinned_empty(n, torch.int32))}
    if kind == "batch":
        offsets = np.concatenate([[0], np.cumsum(_sizes(case))]).astype(np.int32)
        n = int(offsets[-1])
        m = _log_masses(g, n, 1e-7, 1e-4)
        xd, vd = _orbits(g, G * (1.0 + m), _uniform(g, n, 0.1, 5.0), _rayleigh(g, n, 0.02, 0.9), _rayleigh(g, n, 0.01, 1.0))
        x, v, R = _pinned(xd), _pinned(vd), _radii(m).cpu().numpy()
        h = genga.genga_init_batch(offsets, np.ones(case["systems"]), m.cpu().numpy(), R, x, v, G, DT, case["order"], case["steps"])
        return {"case": case, "ctx": _Context(h, x=x, v=v, xo=_pinned_empty((n, 3)), vo=_pinned_empty((n, 3)),
                                              mo=_pinned_empty(n), Ro=_pinned_empty(n), alive=_pinned_empty(n, torch.int32))}
    B, n = case["systems"], case["n"]
    disks = [_disk(g, n) for _ in range(B)]
    m, x, v = (torch.stack([d[k] for d in disks]) for k in range(3))
    normal = lambda: torch.randn(x.shape, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    return {"case": case, "m": m.requires_grad_(), "x": x.requires_grad_(), "v": v.requires_grad_(), "xbar": normal(), "vbar": normal(),
            "engine": adjoint.AdjointEngine(np.ones(B), G, DT, case["order"], case["every"])}


def _ptr(a):
    return a.ctypes.data_as(C.POINTER(C.c_int if a.dtype == np.int32 else C.c_double))


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "kick":
        genga.genga_kick_noalloc(case["n"], G, 3.0, case["kmode"], 0, s["m"], s["alive"], s["x"], s["rc"], s["a"], s["cand"],
                                 len(s["cand"]), s["ncand"])
        return [s["a"], s["cand"], s["ncand"]]
    if kind == "kepler":
        genga.genga_phase_kepler(case["n"], G, DT, 30, s["alive"], s["x"], s["v"], s["fail"])
        return [s["x"], s["v"], s["fail"]]
    if kind == "adjoint":
        xo, vo = adjoint.hybrid_steps(s["x"], s["v"], s["m"], s["engine"], case["steps"])
        gx, gv, gm = torch.autograd.grad((xo, vo), (s["x"], s["v"], s["m"]), (s["xbar"], s["vbar"]))
        return [xo.detach(), vo.detach(), gx, gv, gm]
    c = s["ctx"]
    if kind == "disk":
        genga.genga_set_state(c.handle, c.x, c.v)
        genga.genga_step(c.handle, case["steps"])
        o = genga.genga_get_state(c.handle, case["n"] + 1, **c.out)
        return [o["x"], o["v"], o["m"], o["R"], o["alive"]]
    if kind == "tp":  # goes on from where the last pass left off
        genga.genga_step(c.handle, case["steps"])
        genga._check(genga.lib().genga_get_state_tp(c.handle, _ptr(c.xt), _ptr(c.vt), _ptr(c.alive)), "genga_get_state_tp")
        return [c.xt, c.vt, c.alive]
    genga.genga_set_state_batch(c.handle, c.x, c.v)
    genga.genga_step(c.handle, case["steps"])
    genga._check(genga.lib().genga_get_state_batch(c.handle, _ptr(c.xo), _ptr(c.vo), _ptr(c.mo), _ptr(c.Ro), _ptr(c.alive)),
                 "genga_get_state_batch")
    return [c.xo, c.vo, c.mo, c.Ro, c.alive]


# ------------------------------------------------------------------------------------ work, exact
PAIR = 20.0     # operations of an ordered pair of a kick (sqrt and division as one each)
DRIFT = 250.0   # operations of a body's Kepler drift


def work(case):
    kind = case["kind"]
    if kind == "kick":
        n = case["n"]
        return {"bytes": 8.0 * n * 8, "flops": PAIR * n * (n - 1)}
    if kind == "kepler":
        return {"bytes": 12.0 * 8 * case["n"], "flops": DRIFT * case["n"]}
    sub = case["steps"] * {2: 1, 4: 3, 6: 7}[case["order"]]
    if kind == "disk":
        n = case["n"]
        return {"bytes": (6.0 + 8.0) * 8 * n, "flops": sub * n * (PAIR * (n - 1) + DRIFT)}
    if kind == "tp":
        n = case["n"]
        return {"bytes": 12.0 * 8 * n, "flops": sub * n * (PAIR * case["planets"] + DRIFT)}
    if kind == "batch":  # sizes U{3..63}: mean 33, mean square 1399.7
        s = case["systems"]
        return {"bytes": (6.0 + 8.0) * 8 * 33 * s, "flops": sub * s * (PAIR * (1399.7 - 33) + DRIFT * 33)}
    n, b = case["n"], case["systems"]
    # forward: two kicks a substep; backward: the recomputed forward and its reverse (twice that)
    return {"bytes": (7.0 + 12.0 + 7.0) * 8 * n * b, "flops": 4.0 * sub * b * n * (2 * PAIR * (n - 1) + DRIFT)}


def exact(case, seed):
    """The kick and the drift in plain torch. A simulation's branches (encounter groups, their
    adaptive integration) have no plain closed form: None."""
    if case["kind"] == "kick":
        s = prepare(case, seed)
        x, m, rc = s["x"].T, s["m"], s["rc"]
        d = x[None, :, :] - x[:, None, :]
        r = torch.sqrt((d * d).sum(-1))
        rcij = torch.maximum(rc[:, None], rc[None, :])
        y = ((r - 0.1 * rcij) / (0.9 * rcij)).clamp(0.0, 1.0)
        D = 2.0 * y * y - 2.0 * y + 1.0
        w = y * y / D
        if case["kmode"] == 1:
            w = w - torch.where(y < 1.0, (y + 1.0 / 9.0) * 2.0 * y * (1.0 - y) / (D * D), torch.zeros_like(y))
        f = G * m[None, :] * w / r ** 3
        f.fill_diagonal_(0.0)
        return [(f[:, :, None] * d).sum(1).T.contiguous(), None, None]
    if case["kind"] == "kepler":
        s = prepare(case, seed)
        x, v = s["x"], s["v"]
        r0 = x.norm(dim=0)
        a = 1.0 / (2.0 / r0 - (v * v).sum(0) / G)
        ec, es = 1.0 - r0 / a, (x * v).sum(0) / torch.sqrt(G * a)   # e cos E0, e sin E0
        w = torch.sqrt(G / a ** 3)
        dE = w * DT
        for _ in range(12):  # dM = dE - ec sin dE + es (1 - cos dE)
            f = dE - ec * torch.sin(dE) + es * (1.0 - torch.cos(dE)) - w * DT
            dE = dE - f / (1.0 - ec * torch.cos(dE) + es * torch.sin(dE))
        c1 = 2.0 * torch.sin(0.5 * dE) ** 2                          # 1 - cos dE
        r = a * (1.0 - ec * torch.cos(dE) + es * torch.sin(dE))
        fg, gg = 1.0 - a / r0 * c1, DT - (dE - torch.sin(dE)) / w
        fd, gd = -torch.sqrt(G * a) * torch.sin(dE) / (r * r0), 1.0 - a / r * c1
        return [fg * x + gg * v, fd * x + gd * v, None]
    return None
