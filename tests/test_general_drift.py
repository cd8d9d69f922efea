"""Bound orbits whose steps are too long for the fixed-point solver: the general
solver, from its FP32 start, against the Kepler flow in extended precision."""
import numpy as np
import pytest

from paper_2307_05683_gb300 import inputs
from test_gr_sums import X, drift

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a,e,days", [(0.387, 0.7, 5.0), (0.387, 0.6, 6.5), (1.0, 0.9, 5.0), (5.2, 0.95, 16.0), (1e-4, 0.5, 3e-5),
                                      (0.3, 0.2, 10.0), (1.0, 0.7, 20.0)])
def test_one_long_step_in_extended_precision(a, e, days):
    """Every phase of an orbit whose pericentre timescale is 1.7 to 4 steps: some
    steps are the fixed-point solver's, some the general one's.  The time at
    which the solver stops is wrong by some ten roundings of its terms (about h
    each), so the position by 16 2^-53 of |Q| and of the fastest motion's h v, the
    velocity by the same of v and of the strongest acceleration's h."""
    from paper_2307_05683_gb300 import build, whg
    build.build()
    n = 499
    ens = inputs.test_particle(np.full(n, a), np.full(n, e), np.linspace(0, 2 * np.pi, n, endpoint=False), omega=0.3, inc=0.2,
                               dt=days * inputs.DAY)
    h = float(ens.dt[0])
    first = None
    for S in (n, 12000, 45000):                          # four lanes per planet, few and many warps
        it = whg.Integrator(S, 1, gr_mode=0, queue_steps=0)
        it.init(ens.tile(S))
        it.step(1)
        Q0, v0, _, _ = (x[:n] for x in it.get_raw())
        it.step(1)
        Q1, v1, _, st = (x[:n] for x in it.get_raw())
        it.close()
        assert np.all(st == 0)
        if first is not None:
            assert np.array_equal(Q1, first[0]) and np.array_equal(v1, first[1])
            continue
        first = Q1, v1
        Q, v = drift(X(1), X(h), Q0[:, 0].astype(X), v0[:, 0].astype(X))
        norm = lambda x: np.sqrt((x * x).sum(-1)).astype(float)
        # energy and angular momentum are those of the start: the reference has converged
        en = lambda q, u: (u * u).sum(-1) / 2 - 1 / np.sqrt((q * q).sum(-1))
        assert np.abs(en(Q, v) / en(Q0[:, 0].astype(X), v0[:, 0].astype(X)) - 1).max() < 1e-16
        q = a * (1 - e)
        vmax, amax = np.sqrt((1 + e) / q), 1 / q ** 2
        r, w = norm(Q0[:, 0]), norm(v0[:, 0])
        assert np.all(norm(Q1[:, 0] - Q) <= 16 * 2.0 ** -53 * (r + vmax * h))
        assert np.all(norm(v1[:, 0] - v) <= 16 * 2.0 ** -53 * (w + amax * h))
