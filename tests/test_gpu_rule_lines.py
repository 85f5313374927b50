"""The kernels of default calls on both sides of the sizes where a rule ends, and at sizes whose
shares are summed in several windows (more than 64 source groups), against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_util import (assert_forces_close, assert_types_close, assert_vjp_close, dev,
                      grav_tensors, lib, ljc_tensors, oracle_ljc_system)

pytestmark = pytest.mark.gpu


def _sample(n, count=300):
    idx = np.random.default_rng(n).permutation(n)[:count]
    idx[:4] = 0, 1, n - 2, n - 1
    return np.sort(idx)


# streamed below the line, tiles from it on: 114688, and 163840 without softening or with
# plain sums; 8192 and 12288 are where the variant changes
@pytest.mark.parametrize("n,mode,streamed", [
    (8191, "plain", True), (8192, "plain", True), (114687, "plain", True),
    (114688, "plain", False), (114688, "unsoftened", True), (163839, "unsoftened", True),
    (163840, "unsoftened", False), (163839, "uncompensated", True),
    (163840, "uncompensated", False)])
def test_gravity_lines(n, mode, streamed):
    nb = lib()
    g = workloads.plummer(n, seed=n, eps=0.0 if mode == "unsoftened" else 0.01)
    pos, _ = grav_tensors(g)
    eps = float(np.float32(g.eps))
    comp = mode != "uncompensated"
    # the streamed kernels have no copy of the sources and a slot per row
    tile, js = nb.get_config(nb.LAW_GRAV, n)
    own = nb.workspace_size(n, eps=eps, compensated=comp)
    assert (own != nb.workspace_size(n, eps=eps, compensated=comp, tile=tile, jsplit=js)) == streamed
    assert not streamed or own / (16 * n) > n // 512
    x, _, m = g.f32_as_f64()
    idx = _sample(n)
    ref, phi = oracle.grav_accel(x, m, eps=eps, idx=idx, potential=True)
    for pot in (False, True):
        got = nb.forces(pos, eps=eps, pot=pot, compensated=comp).cpu().numpy()[idx]
        assert_forces_close(got[:, :3], ref, what=f"{mode} {n}")
    e = np.abs(got[:, 3] - phi) / np.abs(phi)
    assert e.max() <= 1e-5


@pytest.mark.parametrize("n", [12289, 40009])
@pytest.mark.parametrize("linear", [False, True])
def test_ljc(n, linear):
    nb = lib()
    s = workloads.ljc_sphere(n, seed=n)
    x, _, m, q, st, et = s.f32_as_f64()
    kq = 332.0637 / (4.0 if linear else 80.0)
    prm = nb.pack_ljc(*(torch.from_numpy(a).to(dev()) for a in (
        q, st[s.types], et[s.types], s.types.astype(np.int32))), kq=kq)
    pos = torch.from_numpy(np.concatenate([x, m[:, None]], 1).astype(np.float32)).to(dev())
    law = nb.LAW_LJC_LINEAR if linear else nb.LAW_LJC
    idx = _sample(n, 700)
    ref, phi = oracle.ljc_force(x, q, st[s.types], et[s.types], kq, idx=idx, potential=True,
                                linear=linear)
    ref = ref / m[idx][:, None]
    for pot in (False, True):
        got = nb.forces(pos, prm, law=law, pot=pot).cpu().numpy()[idx]
        assert_forces_close(got[:, :3], ref, what=f"n={n}")
        # subsets: 16 targets to a block, folded slices
        sub = nb.forces_subset(pos, torch.from_numpy(idx.astype(np.int32)).to(dev()), prm,
                               law=law, pot=pot).cpu().numpy()
        assert_forces_close(sub[:, :3], ref, what=f"subset n={n}")
    for a in (got, sub):
        e = np.abs(a[:, 3] - phi) / np.maximum(np.abs(phi), 1e-3 * np.abs(phi).max())
        assert np.sqrt(np.mean(e * e)) <= 1e-5 and e.max() <= 1e-4


@pytest.mark.parametrize("n", [40009, 131071])
def test_jerk_and_gravity_vjp(n):
    nb = lib()
    g = workloads.plummer(n, seed=n, eps=0.01)
    pos, vel = grav_tensors(g)
    eps = float(np.float32(g.eps))
    x, v, m = g.f32_as_f64()
    idx = _sample(n)
    acc, jerk = nb.forces_jerk(pos, vel, eps=eps)
    ra, rj = oracle.grav_jerk(x, v, m, eps=eps, idx=idx)
    assert_forces_close(acc[:, :3].cpu().numpy()[idx], ra, what=f"acc n={n}")
    assert_forces_close(jerk[:, :3].cpu().numpy()[idx], rj, what=f"jerk n={n}")
    lam = np.random.default_rng(n).standard_normal((n, 4)).astype(np.float32)
    gx, gm, _ = nb.adjoint(pos, torch.from_numpy(lam).to(dev()), eps=eps)
    rg, rm = oracle.grav_vjp(x, m, lam[:, :3].astype(np.float64), eps=eps, idx=idx)
    assert_vjp_close(gx[:, :3].cpu().numpy()[idx], gm.cpu().numpy()[idx], rg, rm, what=f"n={n}")


@pytest.mark.parametrize("linear", [False, True])
def test_ljc_vjp(linear):
    nb = lib()
    n = 20011
    s = workloads.ljc_sphere(n, seed=n)
    pos, _, prm = ljc_tensors(s)
    sysm, x, _ = oracle_ljc_system(s)
    law = nb.LAW_LJC
    if linear:
        _, _, m, q, st, et = s.f32_as_f64()
        kq, law = 332.0637 / 4.0, nb.LAW_LJC_LINEAR
        prm = nb.pack_ljc(*(torch.from_numpy(a).to(dev()) for a in (
            q, st[s.types], et[s.types], s.types.astype(np.int32))), kq=kq)
        sysm = oracle.LJCSystem(m, q, s.types, st, et, kq, linear=True)
    lam = np.random.default_rng(n).standard_normal((n, 4)).astype(np.float32)
    gx, gm, gt = nb.adjoint(pos, torch.from_numpy(lam).to(dev()), prm, law=law)
    rg, rm, rs, re = sysm.vjp(x, lam[:, :3].astype(np.float64))
    assert_vjp_close(gx[:, :3].cpu().numpy(), gm.cpu().numpy(), rg, rm, what=f"n={n}")
    assert_types_close(gt.cpu().numpy(), rs, re, what=f"n={n}")
