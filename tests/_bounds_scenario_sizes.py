"""Run the step kernels of every ensemble size, the work queue and the split
adjoint's tape pool, and print the index-check flags of each context as JSON
(run with WHG_LIBRARY pointing at the debug build; used by
test_large_ensembles.py)."""
import json

import numpy as np
import torch

from paper_2307_05683_gb300 import inputs, whg

flags = {}


def run(name, ens, steps, **kw):
    it = whg.Integrator(ens.n_systems, ens.max_planets, **kw)
    it.init(ens)
    for n in steps:
        it.step(n)
    it.read_state()
    it.energy()
    flags[name] = whg.whg_debug_bounds(it.ctx)
    it.close()


stop = dict(close_encounter_hill=8.0, eject_factor=3.0)
solar, mixed = inputs.solar_ensemble(5, 2600), inputs.compact_ensemble(6, 12000)
run("few_warps", solar, (20,), gr_mode=1)
run("few_warps_mixed", mixed.subset(np.arange(5000)), (60,), gr_mode=2, newton_terms=6, **stop)
run("many_warps", mixed, (30,), gr_mode=1, queue_steps=0)
run("queue", mixed, (60, 45), gr_mode=0, queue_steps=10, block_size=32)
run("queue_stop_repack_graph", mixed, (300,), gr_mode=1, queue_steps=20, block_size=32, repack_frozen=True, steps_per_launch=100,
    graph_launches=2, **stop)
run("four_lanes_mixed", mixed.subset(np.arange(300)), (60,), gr_mode=2, **stop)

dev = lambda a, t=torch.float64: torch.as_tensor(a, dtype=t).cuda().contiguous()
S = 300
ens = mixed.subset(np.arange(S))
it = whg.Integrator(S, 8, gr_mode=1)
whg.whg_init_device(it.ctx, dev(ens.masses), dev(ens.pos), dev(ens.vel), dev(ens.n_planets, torch.int32), dev(ens.dt))
whg.whg_adjoint_schedule(it.ctx, 32, -1)
loss = torch.empty(S, dtype=torch.float64, device="cuda")
whg.whg_adjoint_forward(it.ctx, 230, 50, dev(ens.pos[:, 1:] - ens.pos[:, :1]), loss)
layout = whg.whg_adjoint_layout(it.ctx)
assert layout["chain_sms"] >= 32 and layout["tape_buffers"] == 5, layout
g = [torch.empty((S, 9, 3), dtype=torch.float64, device="cuda") for _ in range(2)]
gm = torch.empty((S, 9), dtype=torch.float64, device="cuda")
for w in (None, dev(np.linspace(0.5, 2.0, S))):
    whg.whg_adjoint_backward(it.ctx, w, *g, gm)
flags["adjoint_split_pool"] = whg.whg_debug_bounds(it.ctx)
it.close()

print(json.dumps(flags))
