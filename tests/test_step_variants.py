"""The step kernels for few and for many warps per SM, and the work queue where it
is used: the same bits."""
import numpy as np
import pytest

from paper_2307_05683_gb300 import inputs

pytestmark = pytest.mark.gpu


def _raw(whg, ens, n, **kw):
    it = whg.Integrator(ens.n_systems, ens.max_planets, **kw)
    it.init(ens)
    it.step(n)
    out = it.read_state() + it.get_raw()
    it.close()
    return out


@pytest.mark.parametrize("gr,nt", [(1, 8), (0, 6), (2, 8)])
@pytest.mark.parametrize("make", [inputs.solar_ensemble, inputs.compact_ensemble])
def test_many_warps_queue_and_few_warps_agree(make, gr, nt):
    """A system's results do not depend on the ensemble around it: an ensemble
    of more than 8 warps per SM (the queue, and plain launches of the kernel
    for many warps) against its first and last 33 systems alone (the kernel for
    few warps)."""
    from paper_2307_05683_gb300 import build, whg
    build.build()
    ens = make(71, 12000 if make is inputs.compact_ensemble else 5600)
    kw = dict(gr_mode=gr, newton_terms=nt)
    many = _raw(whg, ens, 41, queue_steps=0, **kw)
    for u, v in zip(many, _raw(whg, ens, 41, queue_steps=10, **kw)):
        assert np.array_equal(u, v)
    idx = np.r_[0:33, ens.n_systems - 33:ens.n_systems]
    for u, v in zip(many, _raw(whg, ens.subset(idx), 41, **kw)):
        assert np.array_equal(u[idx], v)
