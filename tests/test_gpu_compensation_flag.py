"""compensated=False on the kernels that default calls run: the same bits from direct launches,
jerk and VJPs; plainly added partials from streamed forces, within FP32 rounding."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_util import assert_forces_close, dev, grav_tensors, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1000, 3000, 9000])
def test_flag(n):
    nb = lib()
    g = workloads.plummer(n, seed=n, eps=0.01)
    pos, vel = grav_tensors(g)
    eps = float(np.float32(g.eps))
    idx = torch.arange(0, n, 7, dtype=torch.int32, device=dev())
    pairs = [nb.forces_jerk(pos, vel, eps=eps, compensated=c) +
             nb.adjoint(pos, vel, eps=eps, compensated=c)[:2] +
             (nb.forces_subset(pos, idx, eps=eps, compensated=c),) +
             ((nb.forces(pos, eps=eps, compensated=c),) if n < 4865 else ())
             for c in (True, False)]
    for a, b in zip(*pairs):
        assert torch.equal(a, b)
    if n >= 4865:
        x, _, m = g.f32_as_f64()
        a = nb.forces(pos, eps=eps, compensated=False)
        assert_forces_close(a[:, :3].cpu().numpy(), oracle.grav_accel(x, m, eps=eps))
