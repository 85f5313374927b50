"""Default jerk and gravity VJP of 131072 particles run the block-pair tile of the stored table
(the same bits), whose partial sums take half of the streamed rows'."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_util import assert_forces_close, dev, grav_tensors, lib

pytestmark = pytest.mark.gpu


def test_large_jerk_and_vjp():
    nb = lib()
    n = 131072
    g = workloads.plummer(n, seed=3, eps=0.01)
    pos, vel = grav_tensors(g)
    eps = float(np.float32(g.eps))
    lam = torch.from_numpy(np.random.default_rng(1).standard_normal((n, 4))
                           .astype(np.float32)).to(dev())
    nb.release()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    acc, jerk = nb.forces_jerk(pos, vel, eps=eps)
    gx, gm, _ = nb.adjoint(pos, lam, eps=eps)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 1.6e9
    tile, js = nb.get_config(nb.TABLE_JERK, n)
    for a, b in zip((acc, jerk), nb.forces_jerk(pos, vel, eps=eps, tile=tile, jsplit=js)):
        assert torch.equal(a, b)
    tile, js = nb.get_config(nb.TABLE_VJP_GRAV, n)
    other = nb.adjoint(pos, lam, eps=eps, tile=tile, jsplit=js)
    assert torch.equal(gx, other[0]) and torch.equal(gm, other[1])
    x, _, m = g.f32_as_f64()
    idx = np.arange(0, n, 1501)
    assert_forces_close(acc[:, :3].cpu().numpy()[idx],
                        oracle.grav_accel(x, m, eps=eps, idx=idx.astype(np.int32)))
