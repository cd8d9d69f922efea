"""The step kernels for small ensembles (four lanes per planet), for few and for
many warps per SM, and the work queue where it is used: the same bits."""
import numpy as np
import pytest

from paper_2307_05683_gb300 import inputs
from test_interaction import _inner, _system

pytestmark = pytest.mark.gpu


def _raw(whg, ens, n, **kw):
    it = whg.Integrator(ens.n_systems, ens.max_planets, **kw)
    it.init(ens)
    it.step(1)
    it.step(n - 1)
    out = it.read_state() + it.get_raw()
    it.close()
    return out


@pytest.fixture(scope="module")
def whg():
    from paper_2307_05683_gb300 import build, whg as w
    build.build()
    return w


@pytest.mark.parametrize("gr,nt", [(1, 8), (0, 6), (2, 8)])
@pytest.mark.parametrize("make,mid,large", [(inputs.solar_ensemble, 2600, 5600), (inputs.compact_ensemble, 5000, 12000)])
def test_kernels_for_every_ensemble_size_agree(whg, make, mid, large, gr, nt):
    """A system's results do not depend on the ensemble around it: `large` (more
    than 8 warps per SM: the kernel for many warps, and the queue), its first
    `mid` systems (the kernel for few warps) and its first 33 (four lanes per
    planet)."""
    ens = make(71, large)
    kw = dict(gr_mode=gr, newton_terms=nt)
    many = _raw(whg, ens, 42, queue_steps=0, **kw)
    for u, v in zip(many, _raw(whg, ens, 42, queue_steps=10, **kw)):
        assert np.array_equal(u, v)
    for n in (mid, 33):
        for u, v in zip(many, _raw(whg, ens.subset(np.arange(n)), 42, **kw)):
            assert np.array_equal(u[:n], v)


@pytest.mark.parametrize("gr", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("kind", ["plain", "heavy", "strong", "near", "wide", "massless", "small"])
def test_edges_agree(whg, kind, n, gr):
    """24 systems at the edges of the float-pair form, alone (four lanes per
    planet) and repeated among 20,000 systems of one lane per planet."""
    if n == 1 and kind == "near":
        pytest.skip("needs two planets")
    ens = _system(kind, n, 100 * n + gr)
    kw = dict(gr_mode=gr, c_light=100.0 / np.sqrt(_inner(kind)))
    small = _raw(whg, ens, 30, **kw)
    for u, v in zip(small, _raw(whg, ens.tile(20000), 30, **kw)):
        assert np.array_equal(u, v[:24], equal_nan=True) and np.array_equal(u[:8], v[19992:20000], equal_nan=True)


def test_stop_rules_and_repacking_agree(whg):
    """Both stop rules on 300 compact systems (four lanes per planet, repacked)
    and on the same systems at the head of 12,000."""
    ens = inputs.compact_ensemble(12, 300)
    big = inputs.compact_ensemble(13, 12000)
    for k in ("masses", "pos", "vel", "n_planets", "dt"):
        getattr(big, k)[:300] = getattr(ens, k)
    kw = dict(close_encounter_hill=6.0, eject_factor=3.0, steps_per_launch=10)
    a, b = _raw(whg, ens, 400, **kw), _raw(whg, big, 400, **kw)
    assert (a[2] != 0).sum() >= 5
    for u, v in zip(a, b):
        assert np.array_equal(u, v[:300])


def test_status_bits_with_four_lanes(whg, orc):
    """Unbound, coincident and running systems side by side: the statuses and
    states of the oracle."""
    ens = inputs.two_planet_system(3, 4)
    ens.vel[1, 2] *= 3.0
    ens.pos[2, 2], ens.vel[2, 2] = ens.pos[2, 1], ens.vel[2, 1]
    g = _raw(whg, ens, 50, gr_mode=0)
    o = orc.OracleEnsemble(4, 2, gr_mode=0)
    o.init(ens)
    o.step(50)
    po, vo, so, to = o.read_state()
    assert list(g[2]) == list(so) == [0, 2, 1, 0]
    assert np.abs(g[0] - po).max() <= 1e-12 and np.abs(g[1] - vo).max() <= 1e-12
