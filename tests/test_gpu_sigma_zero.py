"""LJ + Coulomb VJP with atoms without a radius (sigma = 0, as hydrogens of water models): the
sigma and epsilon derivatives are finite and the oracle's, also where the particle count
leaves pads in the kernels' groups."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_util import assert_types_close, assert_vjp_close, dev, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [37, 256, 1000, 2433, 2560, 4097])
@pytest.mark.parametrize("bare", [1, 5])
@pytest.mark.parametrize("linear", [False, True])
def test_sigma_zero(n, bare, linear):
    nb = lib()
    s = workloads.ljc_sphere(n, seed=n)
    rng = np.random.default_rng(n + bare)
    types = (1 + rng.integers(0, 3, n)).astype(np.int32)
    types[rng.permutation(n)[:bare]] = 0
    sig_t = np.array(s.sig_t)
    sig_t[0] = 0.0
    s = dataclasses.replace(s, types=types, sig_t=sig_t)
    x, v, m, q, st, et = s.f32_as_f64()
    kq = 332.0637 / (4.0 if linear else 80.0)
    prm = nb.pack_ljc(*(torch.from_numpy(a).to(dev()) for a in (
        q, st[s.types], et[s.types], s.types)), kq=kq)
    pos = torch.from_numpy(np.concatenate([x, m[:, None]], 1).astype(np.float32)).to(dev())
    lam = rng.standard_normal((n, 4)).astype(np.float32)
    law = nb.LAW_LJC_LINEAR if linear else nb.LAW_LJC
    gx, gm, gt = nb.adjoint(pos, torch.from_numpy(lam).to(dev()), prm, law=law)
    sysm = oracle.LJCSystem(m, q, s.types, st, et, kq, linear=linear)
    rg, rm, rs, re = sysm.vjp(x, lam[:, :3].astype(np.float64))
    assert torch.isfinite(gt).all()
    assert_vjp_close(gx[:, :3].cpu().numpy(), gm.cpu().numpy(), rg, rm, what=f"n={n}")
    assert_types_close(gt.cpu().numpy(), rs, re, what=f"n={n}")
