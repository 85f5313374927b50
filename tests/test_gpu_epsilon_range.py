"""LJ + Coulomb VJP with wells so shallow that 1 / (24 epsilon) leaves FP32's range: the
epsilon derivative (64 bits) is the oracle's."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_util import dev, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 2501])
@pytest.mark.parametrize("eps", [1e-30, 1e-37, 1e-40, 1e-44])
def test_shallow_well(n, eps):
    nb = lib()
    s = workloads.ljc_sphere(n, seed=n)
    x, v, m, q, st, et = s.f32_as_f64()
    et[0] = eps
    kq = 332.0637 / 80.0
    prm = nb.pack_ljc(*(torch.from_numpy(a).to(dev()) for a in (
        q, st[s.types], et[s.types], s.types.astype(np.int32))), kq=kq)
    pos = torch.from_numpy(np.concatenate([x, m[:, None]], 1).astype(np.float32)).to(dev())
    lam = np.random.default_rng(n).standard_normal((n, 4)).astype(np.float32)
    _, _, gt = nb.adjoint(pos, torch.from_numpy(lam).to(dev()), prm, law=nb.LAW_LJC)
    sysm = oracle.LJCSystem(m, q, s.types, st, et, kq)
    _, _, _, re = sysm.vjp(x, lam[:, :3].astype(np.float64))
    got = gt.cpu().numpy()[4:]
    assert np.all(np.isfinite(got))
    np.testing.assert_allclose(got, re, rtol=1e-3)  # FP32 pair terms of both signs
