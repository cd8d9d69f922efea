"""Workloads whose speed is tracked: what users of the library have it do.

Every case is one pass of a user's program through the public calls: initial
conditions on the device -> whg_init_device -> whg_step -> results on the
device (or the allocation-free call, or the adjoint).  `listed` gives the
fixed cases, `draw` further ones of the same ranges, `prepare` the inputs and
the context a program keeps, `run` one pass, `work` its unavoidable bytes and
flops, and `exact` the same results from a plain torch evaluation of the map
in 64 bits.

A case is a dict of plain values:
  call          advance | dense | energy | noalloc | adjoint | autograd
  ens           solar | compact | two_planet | particles (see inputs.py)
  systems, planets (solar: the first n of the 8 planets), steps
  gr_mode, newton_terms, halley_fp32, merge_jumps, stop (both stop rules)
  samples       outputs taken on the way (dense, energy)
  checkpoint    steps per checkpoint (adjoint, autograd)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2307_05683_gb300 import autograd, inputs, whg

_DEFAULTS = {"call": "advance", "ens": "solar", "systems": 1, "planets": 8, "steps": 1, "gr_mode": 1,
             "newton_terms": 8, "halley_fp32": False, "merge_jumps": False, "stop": False, "samples": 1,
             "checkpoint": 100}
_BASE = 4096                    # distinct systems of an ensemble; larger ones repeat them
_HILL, _EJECT = 1.0, 100.0      # stop rules of the uneven ensemble, as the benchmark sets them


def _case(name=None, **kw):
    c = dict(_DEFAULTS, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one Solar System through the allocation-free call, a few steps: latency of the smallest request
        _case("noalloc_one_system", call="noalloc", systems=1, steps=16),
        # ten two-planet systems without GR, as an interactive study runs them: one partly filled warp
        _case("two_planet_10", ens="two_planet", systems=10, planets=2, steps=1000, gr_mode=0),
        # a trajectory of a few hundred systems: the state read out every 10 steps
        _case("dense_output_500", call="dense", systems=500, steps=200, samples=20),
        # an odd count of five-planet systems, GR with the back-reaction, 6-term series
        _case("five_planets_777", systems=777, planets=5, steps=300, gr_mode=2, newton_terms=6),
        # the headline ensemble: 4096 Solar-System-shaped systems, GR on, every option at its default
        _case("solar_4096", systems=4096, steps=1000),
        # the same ensemble with the FP32 start of the Kepler solver switched on
        _case("solar_4096_halley_fp32", systems=4096, steps=600, halley_fp32=True),
        # the energy-error experiment: 2432 systems, the energy taken every 100 steps
        _case("energy_2432", call="energy", systems=2432, steps=500, samples=5),
        # Newtonian planets with the merged jump, between the small and the full GPU
        _case("merged_newtonian_1500", systems=1500, steps=400, gr_mode=0, merge_jumps=True),
        # massless test particles on (a, e) orbits: the drift alone, one planet per system
        _case("particles_20000", ens="particles", systems=20000, planets=1, steps=500, gr_mode=0),
        # compact systems of 2..8 planets with both stop rules: mixed lane groups, frozen systems
        _case("compact_65536", ens="compact", systems=65536, steps=400, stop=True),
        # the largest sweep size: a million systems, a few steps
        _case("solar_2pow20", systems=1 << 20, steps=20),
        # gradients of a final-position loss for a thousand systems, buffers kept as a training loop does
        _case("adjoint_1024", call="adjoint", systems=1024, steps=1000, checkpoint=100),
    ]


def draw(rng):
    """One more case of the listed ones' ranges (rng: random.Random)."""

    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    call = rng.choice(["advance"] * 6 + ["dense", "energy", "noalloc", "adjoint", "autograd"])
    ens = rng.choice(["solar", "solar", "solar", "compact", "two_planet", "particles"])
    planets = 8
    if ens == "solar":
        planets = rng.choice([8, 8, 8, 1, 2, 3, 4, 5, 6, 7])
    elif ens == "two_planet":
        planets = 2
    elif ens == "particles":
        planets = 1
    if call in ("adjoint", "autograd"):
        if ens in ("compact", "particles"):
            ens, planets = "solar", 8
        systems = log_int(1, 1024 if call == "adjoint" else 200)
        steps = log_int(20, 600 if call == "adjoint" else 200)
        return _case(call=call, ens=ens, planets=planets, systems=systems, steps=steps,
                     gr_mode=rng.choice([0, 1, 1, 2]), checkpoint=rng.choice([25, 50, 100, 37]))
    top = {"noalloc": 8192, "dense": 20000, "energy": 20000}.get(call, 1 << 20)
    systems = log_int(1, top)
    steps = max(1, min(log_int(1, 400 if ens == "compact" else 1000), 20_000_000 // systems))
    gr = 0 if ens == "particles" else rng.choice([0, 1, 1, 1, 2])
    kw = {"newton_terms": rng.choice([8, 8, 8, 6]), "halley_fp32": rng.random() < 0.2,
          "merge_jumps": gr == 0 and rng.random() < 0.4, "stop": ens == "compact" and call == "advance"}
    if call in ("dense", "energy"):
        samples = rng.randint(2, 20)
        steps = samples * max(1, min(steps, 400) // samples)
        kw["samples"] = samples
    return _case(call=call, ens=ens, planets=planets, systems=systems, steps=steps, gr_mode=gr, **kw)


# ------------------------------------------------------------- inputs --

def _ensemble(case, seed):
    """The distinct systems of the case (host arrays)."""
    n = min(case["systems"], _BASE)
    if case["ens"] == "solar":
        e = inputs.solar_ensemble(seed, n)
        B = 1 + case["planets"]
        return inputs.Ensemble(e.masses[:, :B].copy(), e.pos[:, :B].copy(), e.vel[:, :B].copy(),
                               np.full(n, case["planets"], np.int32), e.dt)
    if case["ens"] == "compact":
        return inputs.compact_ensemble(seed, n)
    if case["ens"] == "two_planet":
        return inputs.two_planet_system(seed, n)
    rng = np.random.default_rng(seed)            # particles: where the solver is accurate, 5-day steps
    return inputs.test_particle(rng.uniform(0.387, 2.0, n), rng.uniform(0.0, 0.6, n),
                                rng.uniform(0.0, 2 * np.pi, n))


def _device_inputs(case, seed):
    e = _ensemble(case, seed)
    S = case["systems"]
    at = torch.arange(S, device="cuda") % e.n_systems
    dev = lambda a, t=torch.float64: torch.as_tensor(a, dtype=t).cuda()[at].contiguous()
    d = {"m": dev(e.masses), "x": dev(e.pos), "u": dev(e.vel), "n": dev(e.n_planets, torch.int32),
         "dt": dev(e.dt)}
    if case["call"] in ("adjoint", "autograd"):
        off = np.random.default_rng(seed + 7).normal(0.0, 0.05, e.pos[:, 1:].shape)
        d["target"] = dev(e.pos[:, 1:] - e.pos[:, :1] + off)
    return d


def _options(case):
    kw = {"gr_mode": case["gr_mode"], "newton_terms": case["newton_terms"], "halley_fp32": case["halley_fp32"],
          "merge_jumps": case["merge_jumps"]}
    if case["stop"]:
        kw.update(close_encounter_hill=_HILL, eject_factor=_EJECT)
    return kw


def prepare(case, seed):
    S, N = case["systems"], case["planets"]
    st = dict(_device_inputs(case, seed), case=case)
    if case["ens"] != "compact":
        st["n"] = None                           # every system has max_planets planets
    new = lambda *shape, t=torch.float64: torch.empty(shape, dtype=t, device="cuda")
    if case["call"] == "noalloc":
        o = whg.whg_default_options()
        o.gr_mode, o.newton_terms = case["gr_mode"], case["newton_terms"]
        o.halley_fp32, o.merge_jumps = int(case["halley_fp32"]), int(case["merge_jumps"])
        st["options"] = o
    elif case["call"] == "autograd":
        for k in ("m", "x", "u"):
            st[k].requires_grad_()
        return st
    else:
        st["it"] = whg.Integrator(S, N, **_options(case))
    if case["call"] == "adjoint":
        st.update(loss=new(S), gx=new(S, 1 + N, 3), gu=new(S, 1 + N, 3), gm=new(S, 1 + N))
    elif case["call"] == "energy":
        st["E"] = [new(S) for _ in range(case["samples"])]
    else:
        k = case["samples"] if case["call"] == "dense" else 1
        st["out"] = [(new(S, 1 + N, 3), new(S, 1 + N, 3), new(S, t=torch.int32), new(S)) for _ in range(k)]
    return st


def run(st):
    c = st["case"]
    if c["call"] == "noalloc":
        pos, vel, status, t = st["out"][0]
        whg.whg_integrate_noalloc(c["systems"], c["planets"], st["options"], st["m"], st["x"], st["u"], st["n"],
                                  st["dt"], c["steps"], pos, vel, status, t, whg.current_stream())
        return {"pos": pos, "vel": vel, "status": status, "t": t}
    if c["call"] == "autograd":
        loss = autograd.final_position_loss(st["m"], st["x"], st["u"], None, st["dt"], st["target"], c["steps"],
                                            checkpoint_every=c["checkpoint"], gr_mode=c["gr_mode"])
        gm, gx, gu = torch.autograd.grad(loss.sum(), (st["m"], st["x"], st["u"]))
        return {"loss": loss.detach(), "gm": gm, "gx": gx, "gu": gu}
    it = st["it"]
    whg.whg_init_device(it.ctx, st["m"], st["x"], st["u"], st["n"], st["dt"])
    if c["call"] == "adjoint":
        whg.whg_adjoint_forward(it.ctx, c["steps"], c["checkpoint"], st["target"], st["loss"])
        whg.whg_adjoint_backward(it.ctx, None, st["gx"], st["gu"], st["gm"])
        return {"loss": st["loss"], "gm": st["gm"], "gx": st["gx"], "gu": st["gu"]}
    if c["call"] == "energy":
        for E in st["E"]:
            it.step(c["steps"] // c["samples"])
            whg.whg_energy_device(it.ctx, E)
        return {"E": list(st["E"])}
    for pos, vel, status, t in st["out"]:
        it.step(c["steps"] // len(st["out"]))
        whg.whg_read_state_device(it.ctx, pos, vel, status, t)
    if c["call"] == "dense":
        return {"pos": [o[0] for o in st["out"]], "vel": [o[1] for o in st["out"]],
                "status": st["out"][-1][2], "t": st["out"][-1][3]}
    pos, vel, status, t = st["out"][0]
    return {"pos": pos, "vel": vel, "status": status, "t": t}


def work(case):
    """Inputs read once, outputs written once; per system-step the flops of
    the map with Kepler's equation evaluated once at its solution: per planet
    the drift (prologue 20, two 8-term series and the Stiefel functions 42,
    Lagrange coefficients and the new state 34), two jumps 24, the kick's
    update 6, GR 16, and 24 per pair of planets."""
    S, N, T = case["systems"], case["planets"], case["newton_terms"]
    n = 5.0 if case["ens"] == "compact" else float(N)                # mean planet count (2..8)
    pairs = 12.0 if case["ens"] == "compact" else N * (N - 1) / 2    # mean of n (n - 1) / 2 over 2..8
    drift = 54 + 4 * T + 10
    step = n * (drift + 24 + 6 + (16 if case["gr_mode"] else 0)) + 24 * pairs
    state = 8 * S * (1 + N) * 6                                      # positions and velocities
    load = state + 8 * S * (2 + N)
    if case["call"] in ("adjoint", "autograd"):                      # forward, and twice that in reverse
        return {"bytes": load + 8 * S * 3 * N + state + 8 * S * (2 + N), "flops": 3 * S * case["steps"] * step}
    out = {"energy": 8 * S * case["samples"], "dense": state * case["samples"]}.get(case["call"], state)
    return {"bytes": load + out + 12 * S, "flops": S * case["steps"] * step}


# ---------------------------------------------------------- 64-bit values --
# The Wisdom-Holman map in democratic heliocentric coordinates, in plain torch
# float64: Kepler's equation in universal variables solved by Newton steps to
# convergence with 14-term Stumpff series, pairs by broadcasting.

def _stumpff(z, n, terms=14):
    c = torch.full_like(z, 1.0 / math.factorial(n + 2 * terms))
    for k in range(terms - 1, -1, -1):
        c = torch.addcmul(torch.full_like(z, 1.0 / math.factorial(n + 2 * k)), z, c, value=-1.0)
    return c


def _stiefel(beta, X):
    z = beta * X * X
    G2 = X * X * _stumpff(z, 2)
    G3 = X * X * X * _stumpff(z, 3)
    return 1.0 - beta * G2, X - beta * G3, G2, G3


def _drift(q, v, mu, h):
    r0 = (q * q).sum(-1).sqrt()
    eta = (q * v).sum(-1)
    beta = 2.0 * mu / r0 - (v * v).sum(-1)

    def equation(b, e, r, X):
        G0, G1, G2, G3 = _stiefel(b, X)
        return r * G1 + e * G2 + mu * G3 - h, r * G0 + e * G1 + mu * G2

    with torch.no_grad():
        X = h / r0
        for _ in range(8):
            F, dF = equation(beta, eta, r0, X)
            X = X - F / dF
    if q.requires_grad:                          # derivative of the solution: one step with a fixed slope
        F, dF = equation(beta, eta, r0, X)
        X = X - F / dF.detach()
    G0, G1, G2, G3 = _stiefel(beta, X)
    r = (r0 * G0 + eta * G1 + mu * G2).unsqueeze(-1)
    r0, G1, G2, G3, mu = (a.unsqueeze(-1) for a in (r0, G1, G2, G3, mu))
    qn = q - (mu / r0 * G2) * q + (h.unsqueeze(-1) - mu * G3) * v
    vn = v - (mu / (r * r0) * G1) * q - (mu / r * G2) * v
    return qn, vn


def _kick(case, q, v, mp, m0, dt, live):
    d = q.unsqueeze(1) - q.unsqueeze(2)          # [s, i, j] = Q_j - Q_i
    r2 = (d * d).sum(-1)
    same = torch.eye(q.shape[1], dtype=torch.bool, device=q.device)
    r2s = r2.masked_fill(same, 1.0)
    w = (mp.unsqueeze(1) / (r2s * r2s.sqrt())).masked_fill(same, 0.0)
    a = (w.unsqueeze(-1) * d).sum(2)
    if case["gr_mode"]:
        c = inputs.C_LIGHT
        g = -6.0 * (m0 * m0).unsqueeze(-1) * q / (c * c * (q * q).sum(-1).square()).unsqueeze(-1)
        g = g * live.unsqueeze(-1)
        if case["gr_mode"] == 2:
            g = g - (mp.unsqueeze(-1) * g).sum(1, keepdim=True) / m0.unsqueeze(-1)
        a = a + g
    return v + dt.unsqueeze(-1) * a, r2.masked_fill(same, math.inf)


class _Map:
    """The state of the map: heliocentric positions and barycentric velocities."""

    def __init__(self, case, d):
        m, x, u = d["m"], d["x"], d["u"]
        N = case["planets"]
        self.case, self.m0, self.mp, self.dt = case, m[:, :1], m[:, 1:], d["dt"].unsqueeze(1)
        self.live = torch.arange(N, device=m.device).unsqueeze(0) < d["n"].unsqueeze(1)
        self.M = m.sum(1, keepdim=True)
        self.xc = (m.unsqueeze(-1) * x).sum(1) / self.M
        self.vc = (m.unsqueeze(-1) * u).sum(1) / self.M
        park = torch.zeros(N, 3, dtype=m.dtype, device=m.device)
        park[:, 0] = 1e6 * torch.arange(1, N + 1, device=m.device)
        on = self.live.unsqueeze(-1)
        self.q = torch.where(on, x[:, 1:] - x[:, :1], park)
        self.v = torch.where(on, u[:, 1:] - self.vc.unsqueeze(1), torch.zeros_like(park))
        self.n = torch.zeros_like(self.dt)
        self.alive = torch.ones_like(self.dt, dtype=torch.bool)
        self.first = True
        if case["stop"]:
            dx, du = x[:, 1:] - x[:, :1], u[:, 1:] - u[:, :1]
            r = (dx * dx).sum(-1).sqrt()
            a = 1.0 / (2.0 / r - (du * du).sum(-1) / (self.m0 + self.mp))
            a = torch.where(self.live, a, torch.zeros_like(a))
            rh = _HILL * torch.pow((self.mp.unsqueeze(1) + self.mp.unsqueeze(2)) / (3.0 * self.m0.unsqueeze(1)),
                                   1.0 / 3.0) * 0.5 * (a.unsqueeze(1) + a.unsqueeze(2))
            self.near2 = (rh * rh) * (self.live.unsqueeze(1) & self.live.unsqueeze(2))
            self.far2 = (_EJECT * a.amax(1, keepdim=True)) ** 2

    def _jump(self, q, v):
        return q + ((0.5 * self.dt / self.m0).unsqueeze(-1) * (self.mp.unsqueeze(-1) * v).sum(1, keepdim=True))

    def step(self):
        h = 0.5 * self.dt if self.first else self.dt
        self.first = False
        h = h.expand_as(self.mp)
        mu = self.m0.expand_as(self.mp)
        q, v = _drift(self.q, self.v, mu, h)
        q = self._jump(q, v)
        v, r2 = _kick(self.case, q, v, self.mp, self.m0, self.dt, self.live)
        q = self._jump(q, v)
        on = self.live.unsqueeze(-1)
        if self.case["stop"]:
            far = ((self.q * self.q).sum(-1) > self.far2) & self.live
            self.alive = self.alive & ~far.any(1, keepdim=True) & ~(r2 < self.near2).flatten(1).any(1, keepdim=True)
            on = on & self.alive.unsqueeze(-1)
        self.q, self.v = torch.where(on, q, self.q), torch.where(on, v, self.v)
        self.n = self.n + self.alive

    def synced(self):
        mu = self.m0.expand_as(self.mp)
        half = (0.5 * self.dt).expand_as(self.mp)
        q, v = _drift(self.q, self.v, mu, half)
        done = (self.n > 0).unsqueeze(-1)
        return torch.where(done, q, self.q), torch.where(done, v, self.v)

    def inertial(self):
        q, v = self.synced()
        mp, on = self.mp.unsqueeze(-1), self.live.unsqueeze(-1)
        t = self.n * self.dt
        x0 = self.xc + self.vc * t - (mp * q).sum(1) / self.M
        u0 = self.vc - (mp * v).sum(1) / self.m0
        pos = torch.cat([x0.unsqueeze(1), torch.where(on, x0.unsqueeze(1) + q, torch.zeros_like(q))], 1)
        vel = torch.cat([u0.unsqueeze(1), torch.where(on, v + self.vc.unsqueeze(1), torch.zeros_like(v))], 1)
        return pos, vel, t.squeeze(1)

    def energy(self):
        q, v = self.synced()
        d = q.unsqueeze(1) - q.unsqueeze(2)
        r2 = (d * d).sum(-1)
        same = torch.eye(q.shape[1], dtype=torch.bool, device=q.device)
        pair = (self.mp.unsqueeze(1) * self.mp.unsqueeze(2) / r2.masked_fill(same, 1.0).sqrt()).masked_fill(same, 0.0)
        r = (q * q).sum(-1).sqrt()
        E = 0.5 * (self.M * (self.vc * self.vc).sum(-1, keepdim=True)).squeeze(1)
        E = E + (0.5 * self.mp * (v * v).sum(-1) - self.m0 * self.mp / r).sum(1) - 0.5 * pair.flatten(1).sum(1)
        if self.case["gr_mode"]:
            E = E - (3.0 * self.mp * self.m0 ** 2 / (inputs.C_LIGHT ** 2 * r * r)).sum(1)
        p = (self.mp.unsqueeze(-1) * v).sum(1)
        return E + (p * p).sum(-1) / (2.0 * self.m0.squeeze(1))


def exact(case, seed):
    S, steps = case["systems"], case["steps"]
    grads = case["call"] in ("adjoint", "autograd")
    if steps * (25e-3 if grads else 6e-3) + S * steps * 1.5e-6 * (case["planets"] / 8) ** 2 > 60 or (
            grads and S * steps > 1_200_000):
        return None                              # would take too long, or too much memory
    d = _device_inputs(case, seed)
    if grads:
        for k in ("m", "x", "u"):
            d[k].requires_grad_()
        mp = _Map(case, d)
        for _ in range(steps):
            mp.step()
        q, _ = mp.synced()
        loss = ((q - d["target"]) ** 2).sum((1, 2))
        gm, gx, gu = torch.autograd.grad(loss.sum(), (d["m"], d["x"], d["u"]))
        return {"loss": loss.detach(), "gm": gm, "gx": gx, "gu": gu}
    mp = _Map(case, d)
    k = case["samples"] if case["call"] in ("dense", "energy") else 1
    out = []
    for _ in range(k):
        for _ in range(steps // k):
            mp.step()
        out.append(mp.energy() if case["call"] == "energy" else mp.inertial())
    if case["call"] == "energy":
        return {"E": out}
    if case["call"] == "dense":
        return {"pos": [o[0] for o in out], "vel": [o[1] for o in out], "status": None, "t": out[-1][2]}
    pos, vel, t = out[-1]
    return {"pos": pos, "vel": vel, "status": None, "t": t}
