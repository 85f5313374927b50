"""GPU parity of the kernels that default calls of acceleration + jerk, Hermite steps and
force VJPs run (no tile, no j-split): direct launches up to 2432 particles on 152 SMs,
streamed triangle kernels above (rows of 256 targets), at the edges of both, against the
FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_util import (assert_forces_close, assert_types_close, assert_vjp_close, dev,
                      grav_tensors, lib, ljc_tensors, oracle_ljc_system)

pytestmark = pytest.mark.gpu

DIRECT = [1, 2, 7, 9, 257, 1217, 2432]
STREAMED = [2433, 2560, 2561, 4097, 8193]


@pytest.mark.parametrize("n", DIRECT + STREAMED)
@pytest.mark.parametrize("eps", [0.01, 0.0])
def test_jerk_and_gravity_vjp(n, eps):
    nb = lib()
    g = workloads.plummer(n, seed=n, eps=eps)
    pos, vel = grav_tensors(g)
    e = float(np.float32(eps))
    x, v, m = g.f32_as_f64()
    lam = np.random.default_rng(n).standard_normal((n, 4)).astype(np.float32)
    tl = torch.from_numpy(lam).to(dev())
    if n > 1:
        acc, jerk = nb.forces_jerk(pos, vel, eps=e, G=1.3)
        ra, rj = oracle.grav_jerk(x, v, m, eps=e, G=1.3)
        assert_forces_close(acc[:, :3].cpu().numpy(), ra, what=f"acc n={n}")
        assert_forces_close(jerk[:, :3].cpu().numpy(), rj, what=f"jerk n={n}")
        a2, j2 = nb.forces_jerk(pos, vel, eps=e, G=1.3)
        assert torch.equal(acc, a2) and torch.equal(jerk, j2)
    gx, gm, _ = nb.adjoint(pos, tl, eps=e, alpha=0.5)
    if n > 1:
        rg, rm = oracle.grav_vjp(x, m, lam[:, :3].astype(np.float64), eps=e)
        assert_vjp_close(gx[:, :3].cpu().numpy(), gm.cpu().numpy(), 0.5 * rg, 0.5 * rm,
                         what=f"n={n}")
    else:
        assert not gx.any() and not gm.any()
    g2, m2, _ = nb.adjoint(pos, tl, eps=e, alpha=0.5)
    assert torch.equal(gx, g2) and torch.equal(gm, m2)


@pytest.mark.parametrize("n", [1, 3, 257, 1217, 2432, 2433, 2561, 4097])
@pytest.mark.parametrize("linear", [False, True])
def test_ljc_vjp(n, linear):
    nb = lib()
    law = nb.LAW_LJC_LINEAR if linear else nb.LAW_LJC
    s = workloads.ljc_sphere(n, seed=70 + n)
    pos, _, prm = ljc_tensors(s)
    sysm, x, _ = oracle_ljc_system(s)
    if linear:
        _, _, m, q, st, et = s.f32_as_f64()
        kq = 332.0637 / 4.0
        prm = nb.pack_ljc(*(torch.from_numpy(a).to(dev()) for a in (
            q, st[s.types], et[s.types], s.types.astype(np.int32))), kq=kq)
        sysm = oracle.LJCSystem(m, q, s.types, st, et, kq, linear=True)
    lam = np.random.default_rng(n).standard_normal((n, 4)).astype(np.float32)
    tl = torch.from_numpy(lam).to(dev())
    gx, gm, gt = nb.adjoint(pos, tl, prm, law=law)
    g2, m2, t2 = nb.adjoint(pos, tl, prm, law=law)
    assert torch.equal(gx, g2) and torch.equal(gm, m2) and torch.equal(gt, t2)
    if n > 1:
        rg, rm, rs, re = sysm.vjp(x, lam[:, :3].astype(np.float64))
        assert_vjp_close(gx[:, :3].cpu().numpy(), gm.cpu().numpy(), rg, rm, what=f"n={n}")
        assert_types_close(gt.cpu().numpy(), rs, re, what=f"n={n}")
    # the sums over a sweep of two steps, reduced once, are those of two VJPs
    lx, lv = torch.zeros_like(tl), tl.clone()
    gm3 = torch.zeros(n, device=dev())
    gt3 = torch.zeros_like(gt)
    nb.api.adjoint_leapfrog(pos.repeat(2, 1).contiguous(), lx, lv, prm, k=2, dt=1.0, first=False,
                            law=law, G=1.0, eps=0.0, grad_m=gm3, grad_types=gt3, ntypes=4)
    lv4, gt4 = tl.clone(), torch.zeros_like(gt)
    lx4, gm4 = torch.zeros_like(tl), torch.zeros(n, device=dev())
    for step in range(2):
        nb.adjoint(pos, lv4, prm, law=law, grad_x=lx4, grad_m=gm4, grad_types=gt4,
                   accumulate=True)
        lv4[:, :3] += lx4[:, :3]
    assert torch.equal(lx[:, :3], lx4[:, :3])
    np.testing.assert_allclose(gt3.cpu().numpy(), gt4.cpu().numpy(), rtol=1e-12, atol=0)


@pytest.mark.parametrize("n", [300, 2500])
def test_hermite_steps_and_capture(n):
    """k steps in one call are k one-step calls bit for bit, and a captured call replays
    to the eager call's bits."""
    nb = lib()
    pos, vel = grav_tensors(workloads.plummer(n, seed=4, eps=0.01))
    outs = []
    for split in (1, 3):
        p, v = pos.clone(), vel.clone()
        a, j = torch.empty_like(p), torch.empty_like(p)
        for k in range(split):
            nb.hermite_step(p, v, a, j, dt=1e-3, nsteps=3 // split, eps=0.01, acc_valid=k > 0)
        outs.append((p, v, a, j))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    p, v = pos.clone(), vel.clone()
    a, j = torch.empty_like(p), torch.empty_like(p)
    with torch.cuda.stream(side):
        nb.hermite_step(p.clone(), v.clone(), a, j, dt=1e-3, nsteps=3, eps=0.01)
    side.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        nb.hermite_step(p, v, a, j, dt=1e-3, nsteps=3, eps=0.01)
    g.replay()
    torch.cuda.synchronize()
    outs.append((p, v, a, j))
    for other in outs[1:]:
        for s, t in zip(outs[0], other):
            assert torch.equal(s, t)
    nb.sync_check()
