"""GPU parity of the direct kernels (forces on few targets in one launch): small systems,
leapfrog steps and subsets in the library's default configuration, at the edges of their
target groups (8 and 16), source blocks (256), folds (32 blocks) and size rules, against
the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_util import assert_forces_close, dev, grav_tensors, lib

pytestmark = pytest.mark.gpu


def _ljc(n, seed, linear=False):
    nb = lib()
    s = workloads.ljc_sphere(n, seed=seed)
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
    return pos.contiguous(), prm, sysm, x.astype(np.float64)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 16, 17, 255, 256, 257, 1217, 2432, 2433, 4864, 4865])
@pytest.mark.parametrize("mode", ["plain", "pot", "precise", "unsoftened"])
def test_gravity_all(n, mode):
    nb = lib()
    g = workloads.plummer(n, seed=n, eps=0.0 if mode == "unsoftened" else 0.01)
    pos, _ = grav_tensors(g)
    eps = float(np.float32(g.eps))
    x, _, m = g.f32_as_f64()
    a = nb.forces(pos, eps=eps, G=1.7, precise=mode == "precise")
    assert torch.equal(a, nb.forces(pos, eps=eps, G=1.7, precise=mode == "precise"))
    ref, phi = oracle.grav_accel(x, m, G=1.7, eps=eps, potential=True)
    assert_forces_close(a[:, :3].cpu().numpy(), ref, what=f"n={n} {mode}")
    if mode == "pot" and n > 1:
        b = nb.forces(pos, eps=eps, G=1.7, pot=True)
        assert torch.equal(b[:, :3], a[:, :3])
        e = np.abs(b[:, 3].cpu().numpy() - phi) / np.abs(phi)
        assert np.sqrt(np.mean(e * e)) <= 1e-5 and e.max() <= 1e-4


@pytest.mark.parametrize("n", [2, 9, 255, 257, 1217, 2432, 2433])
@pytest.mark.parametrize("linear", [False, True])
def test_ljc_all(n, linear):
    nb = lib()
    law = nb.LAW_LJC_LINEAR if linear else nb.LAW_LJC
    pos, prm, sysm, x = _ljc(n, n, linear)
    a = nb.forces(pos, prm, law=law)
    assert_forces_close(a[:, :3].cpu().numpy(), sysm.accel(x), what=f"n={n}")


@pytest.mark.parametrize("n,na", [(257, 1), (8192, 9), (8193, 300), (40001, 333), (70000, 1500)])
@pytest.mark.parametrize("pot", [False, True])
@pytest.mark.parametrize("law", ["grav", "ljc"])
def test_subset(n, na, pot, law):
    """Active lists in any order, with repeats."""
    nb = lib()
    rng = np.random.default_rng(n + na)
    idx = rng.integers(0, n, na).astype(np.int32)
    idx[-1] = idx[0]
    idx[na // 2] = n - 1
    ti = torch.from_numpy(idx).to(dev())
    if law == "grav":
        g = workloads.plummer(n, seed=n, eps=0.01)
        pos, _ = grav_tensors(g)
        x, _, m = g.f32_as_f64()
        eps = float(np.float32(g.eps))
        a = nb.forces_subset(pos, ti, eps=eps, pot=pot)
        ref, phi = [], []
        for i in idx:  # one target at a time, itself left out
            d = x - x[i]
            r2 = (d * d).sum(1) + eps * eps
            w = m / np.sqrt(r2)
            w[i] = 0.0
            ref.append((d * (w / r2)[:, None]).sum(0))
            phi.append(-w.sum())
        ref, phi = np.array(ref), np.array(phi)
    else:
        if n > 10000:
            pytest.skip("the LJC oracle works on all pairs")
        pos, prm, sysm, x = _ljc(n, n)
        a = nb.forces_subset(pos, ti, prm, pot=pot)
        ref, phi = sysm.accel(x, potential=True)
        ref, phi = ref[idx], phi[idx]
    got = a.cpu().numpy()
    assert_forces_close(got[:, :3], ref, what=f"n={n} na={na}")
    if pot:
        e = np.abs(got[:, 3] - phi) / np.maximum(np.abs(phi), 1e-3 * np.abs(phi).max())
        assert e.max() <= 1e-4
    nb.sync_check()


def test_subset_reports_a_bad_index():
    nb = lib()
    pos, _ = grav_tensors(workloads.plummer(500, seed=1, eps=0.01))
    idx = torch.tensor([3, 500, -1, 4], dtype=torch.int32, device=dev())
    a = nb.forces_subset(pos, idx, eps=0.01)
    with pytest.raises(Exception):
        nb.sync_check()
    good = nb.forces_subset(pos, idx[[0, 3]], eps=0.01)
    nb.sync_check()
    assert torch.equal(a[[0, 3]], good)


@pytest.mark.parametrize("two", [False, True])
@pytest.mark.parametrize("law", ["grav", "ljc"])
@pytest.mark.parametrize("nsteps", [1, 2, 3, 4])
def test_steps(law, two, nsteps):
    """k steps in one call are k one-step calls bit for bit, with the positions of every
    step in the trace, from a fresh and from a carried acceleration, eager and captured;
    masses stay, and forces at the end state have the acceleration's bits."""
    nb = lib()
    n = 777
    if law == "grav":
        pos, vel = grav_tensors(workloads.plummer(n, seed=5, eps=0.01))
        prm, kw, fkw = None, dict(eps=0.01, dt=1e-3), dict(eps=0.01)
    else:
        pos, prm, _, _ = _ljc(n, 5)
        vel, kw, fkw = torch.zeros_like(pos), dict(dt=1e-5), {}
    p, v, a = pos.clone(), vel.clone(), torch.empty_like(pos)
    lo = torch.zeros((2 * n, 4), device=dev()) if two else None
    trace = torch.full(((nsteps + 1) * n, 4), float("nan"), device=dev())
    nb.step(p, v, a, prm, nsteps=nsteps, state_lo=lo, trace=trace, **kw)
    q, w, b = pos.clone(), vel.clone(), torch.empty_like(pos)
    lo2 = torch.zeros((2 * n, 4), device=dev()) if two else None
    for k in range(nsteps):
        assert torch.equal(trace[k * n:(k + 1) * n], q)
        nb.step(q, w, b, prm, nsteps=1, acc_valid=k > 0, state_lo=lo2, **kw)
    assert torch.equal(trace[nsteps * n:], q)
    for s, t in ((p, q), (v, w), (a, b)):
        assert torch.equal(s[:, :3], t[:, :3])
    assert not two or torch.equal(lo, lo2)
    assert torch.equal(p[:, 3], pos[:, 3])
    assert torch.equal(nb.forces(p, prm, **fkw)[:, :3], a[:, :3])
    # reported steps leave the same state, and rows that calls of one step report
    q, w, b = pos.clone(), vel.clone(), torch.empty_like(pos)
    lo2 = torch.zeros((2 * n, 4), device=dev()) if two else None
    rows = nb.step(q, w, b, prm, nsteps=nsteps, report_every=2, state_lo=lo2, **kw)
    for s, t in ((p, q), (v, w), (a, b)):
        assert torch.equal(s[:, :3], t[:, :3])
    assert rows.shape[0] == nsteps // 2 + 1
    hi, rest = nb.forces(q, prm, want_lo=True, **fkw)
    assert torch.equal(hi[:, :3], a[:, :3])
    assert float(rest.abs().max()) <= float(hi.abs().max()) * 2 ** -23
    # the carried acceleration, all steps in one call, and the same call captured
    outs = []
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    for captured in (False, True):
        q, w, b = pos.clone(), vel.clone(), torch.empty_like(pos)
        lo2 = torch.zeros((2 * n, 4), device=dev()) if two else None
        with torch.cuda.stream(side):
            nb.step(q, w, b, prm, nsteps=1, state_lo=lo2, **kw)
            if captured:
                g = torch.cuda.CUDAGraph()
                side.synchronize()
        if captured:
            with torch.cuda.graph(g, stream=side):
                nb.step(q, w, b, prm, nsteps=nsteps, acc_valid=True, state_lo=lo2, **kw)
            g.replay()
        else:
            with torch.cuda.stream(side):
                nb.step(q, w, b, prm, nsteps=nsteps, acc_valid=True, state_lo=lo2, **kw)
        torch.cuda.synchronize()
        outs.append((q, w, b) + ((lo2,) if two else ()))
    for s, t in zip(*outs):
        assert torch.equal(s[:, :3], t[:, :3])
    if nsteps > 1:  # one step, then nsteps more: a call of nsteps + 1
        q, w, b = pos.clone(), vel.clone(), torch.empty_like(pos)
        lo2 = torch.zeros((2 * n, 4), device=dev()) if two else None
        nb.step(q, w, b, prm, nsteps=nsteps + 1, state_lo=lo2, **kw)
        assert torch.equal(q, outs[0][0]) and torch.equal(w[:, :3], outs[0][1][:, :3])
    nb.sync_check()


def test_output_over_the_positions():
    """Accelerations written over the positions they come from: still the general path's
    answer (a direct launch would read what it has overwritten)."""
    nb = lib()
    pos, _ = grav_tensors(workloads.plummer(900, seed=8, eps=0.01))
    want = nb.forces(pos, eps=0.01)
    over = pos.clone()
    nb.forces(over, eps=0.01, out=over)
    np.testing.assert_allclose(over[:, :3].cpu().numpy(), want[:, :3].cpu().numpy(), rtol=1e-4,
                               atol=1e-6 * float(want.abs().max()))
