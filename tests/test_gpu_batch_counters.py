"""A plan's captured run stays valid when a later run needs more work counters."""
import pytest
import torch

import workloads
from gpu_util import grav_tensors, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [-1, 0])
def test_graph_after_a_longer_run(tile):
    nb = lib()
    table, at, parts = [], 0, []
    for n in (900, 64, 1501):
        parts.append(grav_tensors(workloads.plummer(n, seed=n, eps=0.01)))
        table.append(dict(offset=at, n=n, law=nb.LAW_GRAV, eps=0.01, dt=1e-3))
        at += n
    pos, vel = (torch.cat([p[c] for p in parts]) for c in (0, 1))
    outs = []
    for graph in (True, False):
        plan = nb.BatchPlan(table, tile=tile)
        p, v, a = pos.clone(), vel.clone(), torch.zeros_like(pos)
        plan.run(p, v, a, nsteps=0, graph=False)
        for steps, captured in ((5, graph), (20, False), (5, graph), (40, False), (5, graph)):
            plan.run(p, v, a, nsteps=steps, acc_valid=True, graph=captured)
            torch.cuda.synchronize()
            held = torch.full((1 << 20,), 7, dtype=torch.int32, device=p.device)
            del held
        outs.append((p, v, a))
        plan.close()
    for s, t in zip(*outs):
        assert torch.equal(s, t)
    nb.sync_check()
