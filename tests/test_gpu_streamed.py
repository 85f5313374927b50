"""GPU parity of the streamed triangle kernels that default calls run (no tile, no
j-split): sizes around the edges of their rows (256, 384 and 512 targets), source groups
(32) and variants (a change of row length at 12288 and 32768), against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_util import assert_forces_close, dev, grav_tensors, lib, oracle_ljc_system

pytestmark = pytest.mark.gpu

SIZES = [2500, 2559, 2560, 2561, 3071, 3073, 4097, 8191, 12287, 12288, 12289]


@pytest.mark.parametrize("n", SIZES + [32767, 32768])
@pytest.mark.parametrize("mode", ["plain", "pot", "precise", "uncompensated", "unsoftened"])
def test_gravity(n, mode):
    nb = lib()
    if n > 12289 and mode not in ("plain", "pot"):
        pytest.skip("the large variant is the same code")
    g = workloads.plummer(n, seed=n, eps=0.0 if mode == "unsoftened" else 0.01)
    pos, _ = grav_tensors(g)
    eps = float(np.float32(g.eps))
    x, _, m = g.f32_as_f64()
    kw = dict(pot=mode == "pot", precise=mode == "precise",
              compensated=mode != "uncompensated")
    a = nb.forces(pos, eps=eps, G=1.7, **kw)
    assert torch.equal(a, nb.forces(pos, eps=eps, G=1.7, **kw))
    ref, phi = oracle.grav_accel(x, m, G=1.7, eps=eps, potential=True)
    got = a.cpu().numpy()
    assert_forces_close(got[:, :3], ref, what=f"n={n} {mode}")
    if mode == "pot":
        e = np.abs(got[:, 3] - phi) / np.abs(phi)
        assert np.sqrt(np.mean(e * e)) <= 1e-5 and e.max() <= 1e-4
    # the pair term is applied to both particles: momentum is kept to FP32 rounding
    p = np.abs((m[:, None] * got[:, :3].astype(np.float64)).sum(0))
    assert np.all(p <= 1e-6 * np.sum(m[:, None] * np.abs(got[:, :3]), 0))
    hi, lo = nb.forces(pos, eps=eps, G=1.7, want_lo=True)
    if mode == "plain":
        assert torch.equal(hi, a) and float(lo.abs().max()) <= float(hi.abs().max()) * 2 ** -23


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("linear", [False, True])
def test_ljc(n, linear):
    nb = lib()
    law = nb.LAW_LJC_LINEAR if linear else nb.LAW_LJC
    s = workloads.ljc_sphere(n, seed=n)
    x, v, m, q, st, et = s.f32()
    d = dev()
    kq = 332.0637 / (4.0 if linear else 80.0)
    pos = torch.from_numpy(np.concatenate([x, m[:, None]], 1).astype(np.float32)).to(d)
    prm = nb.pack_ljc(torch.from_numpy(q.astype(np.float64)).to(d),
                      torch.from_numpy(st.astype(np.float64)[s.types]).to(d),
                      torch.from_numpy(et.astype(np.float64)[s.types]).to(d),
                      torch.from_numpy(s.types).to(d), kq=kq)
    sysm = oracle.LJCSystem(m.astype(np.float64), q.astype(np.float64), s.types,
                            st.astype(np.float64), et.astype(np.float64), kq, linear=linear)
    ref, phi = sysm.accel(x.astype(np.float64), potential=True)
    a = nb.forces(pos.contiguous(), prm, law=law, pot=True)
    assert torch.equal(a, nb.forces(pos.contiguous(), prm, law=law, pot=True))
    got = a.cpu().numpy()
    assert_forces_close(got[:, :3], ref, what=f"n={n}")
    e = np.abs(got[:, 3] - phi) / np.maximum(np.abs(phi), 1e-3 * np.abs(phi).max())
    assert np.sqrt(np.mean(e * e)) <= 1e-5 and e.max() <= 1e-4
    plain = nb.forces(pos.contiguous(), prm, law=law)
    assert_forces_close(plain[:, :3].cpu().numpy(), ref, what=f"n={n} without potential")


@pytest.mark.parametrize("law", ["grav", "ljc"])
def test_steps_and_capture(law):
    """k steps in one call are k one-step calls bit for bit (with the diagnostics rows),
    and a captured call replays to the eager call's bits."""
    nb = lib()
    n = 3100
    if law == "grav":
        g = workloads.plummer(n, seed=5, eps=0.01)
        pos, vel = grav_tensors(g)
        prm, kw = None, dict(eps=float(np.float32(g.eps)), dt=1e-3)
    else:
        s = workloads.ljc_sphere(n, seed=5)
        x, v, m, q, st, et = s.f32()
        d = dev()
        pos = torch.from_numpy(np.concatenate([x, m[:, None]], 1).astype(np.float32)).to(d)
        vel = torch.zeros_like(pos)
        prm = nb.pack_ljc(torch.from_numpy(q.astype(np.float64)).to(d),
                          torch.from_numpy(st.astype(np.float64)[s.types]).to(d),
                          torch.from_numpy(et.astype(np.float64)[s.types]).to(d),
                          torch.from_numpy(s.types).to(d))
        kw = dict(dt=1e-5)
    runs = []
    for split in (False, True):
        p, w, a = pos.clone().contiguous(), vel.clone().contiguous(), torch.empty_like(pos)
        lo = torch.zeros((2 * n, 4), device=dev())
        if split:
            nb.step(p, w, a, prm, nsteps=1, state_lo=lo, **kw)
            for _ in range(3):
                nb.step(p, w, a, prm, nsteps=1, acc_valid=True, state_lo=lo, **kw)
        else:
            nb.step(p, w, a, prm, nsteps=4, report_every=2, state_lo=lo, **kw)
        runs.append((p, w, a, lo))
    for u, w in zip(*runs):  # acc.w: the potential, on report steps only
        assert torch.equal(u[:, :3], w[:, :3])
    p, w, a = pos.clone().contiguous(), vel.clone().contiguous(), torch.empty_like(pos)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        nb.step(p.clone(), w.clone(), a.clone(), prm, nsteps=2, **kw)  # sizes the workspace
    side.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        nb.step(p, w, a, prm, nsteps=2, **kw)
    g.replay()
    torch.cuda.synchronize()
    p2, w2, a2 = pos.clone().contiguous(), vel.clone().contiguous(), torch.empty_like(pos)
    nb.step(p2, w2, a2, prm, nsteps=2, **kw)
    assert torch.equal(p, p2) and torch.equal(w, w2) and torch.equal(a, a2)
    nb.sync_check()


def test_installed_tile_is_preferred():
    """An entry that the caller installs is run (and gives the tile's bits); a stored one
    leaves the call with the streamed kernel."""
    nb = lib()
    g = workloads.plummer(3000, seed=6, eps=0.01)
    pos, _ = grav_tensors(g)
    base = nb.forces(pos, eps=0.01)
    tile, js = 8, 2
    explicit = nb.forces(pos, eps=0.01, tile=tile, jsplit=js)
    assert not torch.equal(base, explicit)
    old = nb.get_config(nb.LAW_GRAV, 3000)
    raw = nb._lib.load()
    try:
        nb.set_tuned(nb.LAW_GRAV, 3000, tile, js)
        assert torch.equal(nb.forces(pos, eps=0.01), explicit)
        assert raw.nbody_set_stored(nb.LAW_GRAV, 11, tile, js) == 0
        assert nb.get_config(nb.LAW_GRAV, 3000) == (tile, js)
        assert torch.equal(nb.forces(pos, eps=0.01), base)
    finally:
        raw.nbody_set_stored(nb.LAW_GRAV, 11, *old)
