"""Ensembles above 8 warps per SM, where launches of several units run on the
work queue, and the adjoint schedules that small and large ensembles take:
the same bits as plain launches and as each other."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2307_05683_gb300 import inputs

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def whg():
    from paper_2307_05683_gb300 import build, whg as w
    build.build()
    return w


def _many_warps(ens):
    """Whether the default packing (one lane per planet) has more than 8 warps per SM."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per_warp = 32 // np.arange(1, 9)
    counts = np.bincount(ens.n_planets, minlength=9)[1:]
    return int((-(-counts // per_warp)).sum()) > 8 * sms


def _outputs(whg, ens, steps, **kw):
    it = whg.Integrator(ens.n_systems, ens.max_planets, **kw)
    it.init(ens)
    for n in steps:
        it.step(n)
    out = it.read_state() + it.get_raw() + (it.energy(),)
    it.close()
    return out


def _same(a, b):
    return all(np.array_equal(x, y, equal_nan=x.dtype.kind == "f") for x, y in zip(a, b))


@pytest.mark.parametrize("extra", [{}, {"graph_launches": 3, "steps_per_launch": 150},
                                   {"repack_frozen": True, "steps_per_launch": 100}])
def test_queue_with_stop_rules_graphs_and_repacking(whg, extra):
    """Mixed planet counts, both stop rules (many systems stop on the way), units
    of 37 and 25 steps, two calls."""
    ens = inputs.compact_ensemble(46, 12000)
    assert _many_warps(ens)
    kw = dict(close_encounter_hill=8.0, eject_factor=3.0, block_size=32, **extra)
    plain = _outputs(whg, ens, (500, 160), queue_steps=0, **kw)
    assert 200 < int((plain[2] != 0).sum()) < 11800
    for unit in (37, 25):
        assert _same(plain, _outputs(whg, ens, (500, 160), queue_steps=unit, **kw)), unit


@pytest.mark.parametrize("S", [3, 300, 1500, 2500, 5000, 7000, 12000])
@pytest.mark.parametrize("extra", [{}, {"graph_launches": 3, "steps_per_launch": 20, "close_encounter_hill": 8.0,
                                        "gr_mode": 2, "newton_terms": 6}])
def test_blocks_for_several_planet_counts(whg, S, extra):
    """Automatic blocks of 1 to 8 warps (several lane-group sizes in an ensemble,
    block borders inside buckets and across them) against one-warp blocks, and
    the queue, which they replace up to 128 warps per SM."""
    ens = inputs.compact_ensemble(47, S)
    one = _outputs(whg, ens, (90, 410), block_size=32, **extra)
    assert _same(one, _outputs(whg, ens, (90, 410), **extra))
    assert _same(one, _outputs(whg, ens, (90, 410), block_size=160, queue_steps=0, **extra))


def test_queue_units_and_short_launches(whg):
    """Below 4 units a plain launch, a partial last unit, one-step units; then a
    queue whose every wait ran out is used again."""
    ens = inputs.solar_ensemble(49, 5600)
    assert _many_warps(ens)
    steps = (30, 45, 40, 4)
    plain = _outputs(whg, ens, steps, queue_steps=0)
    for unit in (10, 1):
        assert _same(plain, _outputs(whg, ens, steps, queue_steps=unit)), unit
    it = whg.Integrator(5600, 8, queue_steps=10)
    it.init(ens)
    assert whg.whg_test_queue_timeout(it.ctx, 1 << 12) == 1
    it.synchronize()
    for n in steps:
        it.step(n)
    it.synchronize()
    got = it.read_state()
    it.close()
    assert _same(plain, got)


def _gradients(whg, ens, target, n, K, schedule=None, twice=False, keep=None):
    import torch
    dev = lambda a, t=torch.float64: torch.as_tensor(a, dtype=t).cuda().contiguous()
    S, N = ens.n_systems, ens.max_planets
    it = keep or whg.Integrator(S, N, gr_mode=1)
    whg.whg_init_device(it.ctx, dev(ens.masses), dev(ens.pos), dev(ens.vel), dev(ens.n_planets, torch.int32), dev(ens.dt))
    if schedule:
        whg.whg_adjoint_schedule(it.ctx, *schedule)
    loss = torch.empty(S, dtype=torch.float64, device="cuda")
    whg.whg_adjoint_forward(it.ctx, n, K, dev(target), loss)
    out = [loss.cpu().numpy()]
    for w in (None, dev(np.linspace(0.5, 2.0, 2000)[:S])) if twice else (None,):
        g = [torch.empty((S, 1 + N, 3), dtype=torch.float64, device="cuda") for _ in range(2)]
        g.append(torch.empty((S, 1 + N), dtype=torch.float64, device="cuda"))
        whg.whg_adjoint_backward(it.ctx, w, *g)
        out += [x.cpu().numpy() for x in g]
    it.synchronize()
    layout = whg.whg_adjoint_layout(it.ctx)
    if not keep:
        it.close()
    return out, layout


@pytest.mark.parametrize("make", [inputs.solar_ensemble, inputs.compact_ensemble])
def test_adjoint_of_small_ensembles_agrees_with_large_ones(whg, make):
    """The last tapes beside the forward half (ensembles of few warps) against
    all tapes in the backward half (1500 and more systems, unsplit): fewer, as
    many and more segments than tape buffers, a partial last one, a second
    backward call with weights, every schedule, and one context for all."""
    big = make(91, 2000)
    target = big.pos[:, 1:] - big.pos[:, :1] + 0.01
    small = big.subset(np.arange(60))
    it = whg.Integrator(60, 8, gr_mode=1)
    for n in (30, 100, 150, 230):
        ref, layout = _gradients(whg, big, target, n, 50, (0, 0), True)
        assert layout["chain_sms"] == 0
        for schedule in ((-1, 0), (0, 0), (-1, -1), (16, 0), (16, -1)):
            got, layout = _gradients(whg, small, target[:60], n, 50, schedule, True, it)
            assert (layout["chain_sms"] > 0) == (schedule[0] > 0)
            for a, b in zip(ref, got):
                assert np.array_equal(a[:60], b, equal_nan=True), (n, schedule)
    it.close()


def test_debug_build_index_checks_of_every_step_kernel():
    """tests/_bounds_scenario_sizes.py with the index checks compiled in."""
    from paper_2307_05683_gb300 import build
    lib = build.build(debug=True)
    env = dict(os.environ, WHG_LIBRARY=lib, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "_bounds_scenario_sizes.py")], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    flags = json.loads(r.stdout.strip().splitlines()[-1])
    assert len(flags) == 7 and all(v == 0 for v in flags.values()), flags
