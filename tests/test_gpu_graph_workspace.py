"""A captured call keeps its workspace when later calls on the same stream need a larger one."""
import pytest
import torch

import workloads
from gpu_util import grav_tensors, lib

pytestmark = pytest.mark.gpu


def test_replay_after_growth():
    nb = lib()
    sizes = (5001, 20001, 60001)
    side = torch.cuda.Stream()
    runs = []
    for n in sizes:
        pos, vel = grav_tensors(workloads.plummer(n, seed=n, eps=0.01))
        acc = nb.forces(pos, eps=0.01)
        want = [t.clone() for t in (pos, vel, acc)]
        for _ in range(2):
            nb.step(*want, dt=1e-3, nsteps=3, eps=0.01, acc_valid=True)
        torch.cuda.synchronize()
        with torch.cuda.stream(side):  # sizes the workspace of this stream
            nb.forces(pos.clone(), eps=0.01)
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            nb.step(pos, vel, acc, dt=1e-3, nsteps=3, eps=0.01, acc_valid=True)
        runs.append((graph, (pos, vel, acc), want))
    big, _ = grav_tensors(workloads.plummer(100000, seed=1, eps=0.01))
    with torch.cuda.stream(side):
        nb.forces(big, eps=0.01)
    for _ in range(2):
        for graph, _, _ in runs:
            graph.replay()
    torch.cuda.synchronize()
    for _, got, want in runs:
        for a, b in zip(got, want):
            assert torch.equal(a, b)
    nb.sync_check()
    del runs
    nb.release()
