"""Strong GR terms and heavy planets: one step of every step kernel against the
map in extended precision."""
import numpy as np
import pytest

from paper_2307_05683_gb300 import inputs

pytestmark = pytest.mark.gpu

X = np.longdouble


def stiefel(beta, s):
    z = beta * s * s
    out = []
    for n in (2, 3):
        c = np.zeros_like(z)
        for k in range(14, -1, -1):                      # (-z)^k / (n + 2k)!, nested
            c = (1 - z * c) / X((n + 2 * k) * (n + 2 * k - 1)) if k else 1 - z * c
        out.append(c / X([2, 6][n - 2]))
    G2, G3 = s * s * out[0], s ** 3 * out[1]
    return 1 - beta * G2, s - beta * G3, G2, G3


def drift(mu, h, q, v):
    """The Kepler flow (universal variables, Newton steps to convergence)."""
    r0, eta = np.sqrt((q * q).sum(-1)), (q * v).sum(-1)
    beta = 2 * mu / r0 - (v * v).sum(-1)
    s = h / r0
    for _ in range(30):
        G0, G1, G2, G3 = stiefel(beta, s)
        s = s - (r0 * G1 + eta * G2 + mu * G3 - h) / (r0 * G0 + eta * G1 + mu * G2)
    G0, G1, G2, G3 = stiefel(beta, s)
    r = r0 * G0 + eta * G1 + mu * G2
    e = lambda a: a[..., None]
    return (q - e(mu / r0 * G2) * q + e(h - mu * G3) * v, v - e(mu / (r * r0) * G1) * q - e(mu / r * G2) * v)


def step(m0, m, dt, c, gr, Q, v):
    """One step with a whole drift, Q and v [S, n, 3]."""
    m0, m, dt, Q, v = (np.asarray(a, X) for a in (m0, m, dt, Q, v))
    e = lambda a: a[..., None]
    Q, v = drift(e(m0) + 0 * m, e(dt) + 0 * m, Q, v)
    jump = lambda: e(e(dt / (2 * m0))) * (e(m) * v).sum(1, keepdims=True)
    Q = Q + jump()
    d = Q[:, None] - Q[:, :, None]                       # [s, i, j] = Q_j - Q_i
    r2 = (d * d).sum(-1)
    w = np.where(r2 == 0, X(0), m[:, None] / np.where(r2 == 0, X(1), r2) ** X(1.5))
    a = (e(w) * d).sum(2)
    g = -6 * e(e(m0 * m0)) * Q / (X(c) ** 2 * e((Q * Q).sum(-1) ** 2))
    if gr == 2:
        g = g - (e(m) * g).sum(1, keepdims=True) / e(e(m0))
    v = v + e(e(dt)) * (a + (g if gr else 0))
    return Q + jump(), v


def _systems(n, m_heavy, ratio, heavy, seed, S=6):
    rng = np.random.default_rng(seed)
    a = 0.05 * float(ratio) ** np.arange(n) * np.ones((S, 1))
    m = 10.0 ** rng.uniform(-8, -5, (S, n))
    m[:, heavy] = m_heavy * rng.uniform(0.8, 1.0, S)
    ang = rng.uniform(0, 2 * np.pi, (3, S, n))
    x, v = inputs.elements_to_state(1.0 + m, a, rng.uniform(0, 0.05, (S, n)), rng.uniform(0, 0.05, (S, n)), *ang)
    return inputs._assemble(1.0, m, x, v, np.full(S, n), 2 * np.pi * np.sqrt(a[:, 0] ** 3) / 25, "strong GR")


@pytest.mark.parametrize("gr", [1, 2])
@pytest.mark.parametrize("light", [60.0, 300.0, 3000.0, 1e5])
@pytest.mark.parametrize("m_heavy,ratio,n,heavy", [(1e-9, 1.7, 8, 0), (1e-3, 1.7, 8, 0), (1e-3, 1.7, 5, 0), (1e-3, 1.7, 6, 5),
                                                   (1e-3, 2.0, 4, 0), (0.02, 8.0, 4, 0), (0.02, 8.0, 2, 1), (0.05, 12.0, 2, 0),
                                                   (1e-3, 1.7, 1, 0), (0.3, 1.7, 1, 0)])
def test_one_step_in_extended_precision(m_heavy, ratio, n, heavy, light, gr):
    """The light speed is `light` orbital speeds of the innermost planet (GR kicks
    of 2^-11 to 2^-33 of its velocity).  A coordinate of Q or v takes some ten
    roundings in a step, none of a value much above the planet's own |Q| or
    |v|: 2^-49 of those bounds them; a sum in 24 bits shows up to 2^-36."""
    from paper_2307_05683_gb300 import build, whg
    build.build()
    ens = _systems(n, m_heavy, ratio, heavy, 1000 * n + int(10 * ratio) + heavy)
    c = light / np.sqrt(0.05)
    for S in (6, {1: 12000, 2: 8000}.get(n, 2600), 40000 if n < 4 else 12000):     # four lanes per planet, few and many warps
        big = ens.tile(S)
        it = whg.Integrator(S, n, gr_mode=gr, c_light=c, queue_steps=0)
        it.init(big)
        it.step(1)
        Q0, v0, _, _ = it.get_raw()
        it.step(1)
        Q1, v1, _, st = it.get_raw()
        it.close()
        assert np.all(st == 0)
        Q, v = step(ens.masses[:, 0], ens.masses[:, 1:], ens.dt, c, gr, Q0[:6], v0[:6])
        norm = lambda a: np.sqrt((a * a).sum(-1))
        eq, ev = norm(Q1[:6] - Q) / norm(Q), norm(v1[:6] - v) / norm(v)
        assert eq.max() <= 2.0 ** -49 and ev.max() <= 2.0 ** -49, (S, np.log2(float(eq.max())), np.log2(float(ev.max())))
        assert np.array_equal(Q1[:6], Q1[S - S % 6 - 6:S - S % 6]) and np.array_equal(v1[:6], v1[S - S % 6 - 6:S - S % 6])
