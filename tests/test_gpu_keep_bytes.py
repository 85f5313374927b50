"""leapfrog(keep_bytes=0) holds what its checkpoints take, and gives the same gradients."""
import numpy as np
import pytest
import torch

import workloads
from gpu_util import dev, lib

pytestmark = pytest.mark.gpu


def test_footprint_and_gradients():
    nb = lib()
    from paper_0706_3060_gb300.autograd import leapfrog
    n, nsteps, k = 20000, 150, 10
    x, v, m = workloads.plummer(n, seed=1, eps=0.01).f32()
    w = torch.from_numpy(np.random.default_rng(3).standard_normal((2, n, 3))
                         .astype(np.float32)).to(dev())
    outs, held = [], []
    for keep in (0, None):
        leaves = [torch.from_numpy(np.ascontiguousarray(a)).to(dev()).requires_grad_(True)
                  for a in (x, v, m)]
        torch.cuda.synchronize()
        before = torch.cuda.memory_allocated()
        xT, vT = leapfrog(*leaves, nsteps=nsteps, k=k, dt=1e-4, eps=0.01, keep_bytes=keep)
        held.append(torch.cuda.memory_allocated() - before)
        outs.append(torch.autograd.grad([xT, vT], leaves, [w[0], w[1]]))
        del xT, vT
    for a, b in zip(*outs):
        assert torch.equal(a, b)
    rows = 5 * (nsteps // k) + k + 1 + 3  # checkpoints, newest positions, x_T, v_T and pos
    assert held[0] <= (rows + 1) * 16 * n
    assert held[1] >= nsteps * 16 * n  # 48 MB: kept on an empty device
    nb.sync_check()
