"""Calls of several steps on arrays that start 16 bytes past a cache line: the same bits as
one-step calls. There a line of positions, velocities or lambda is written by two blocks of
the finalize, while the next evaluation's kernel, placed early, waits to read it."""
import numpy as np
import pytest
import torch

import workloads
from gpu_util import dev, grav_tensors, lib, ljc_tensors

pytestmark = pytest.mark.gpu


def _shifted(t):
    """A copy of t that starts 16 bytes past a multiple of 128."""
    out = torch.empty(t.numel() + 64, dtype=t.dtype, device=t.device)
    skip = (-out.data_ptr() % 128 + 16) // 4
    out = out[skip:skip + t.numel()].view(t.shape)
    assert out.data_ptr() % 128 == 16
    return out.copy_(t)


def _system(law, n):
    nb = lib()
    if law == "grav":
        pos, vel = grav_tensors(workloads.plummer(n, seed=n, eps=0.01))
        return _shifted(pos), _shifted(vel), None, dict(eps=0.01)
    pos, vel, prm = ljc_tensors(workloads.ljc_sphere(n, seed=n))
    return _shifted(pos), _shifted(vel), _shifted(prm), dict(law=nb.LAW_LJC)


def _same(outs):
    for s, t in zip(*outs):
        assert torch.equal(s, t)


@pytest.mark.parametrize("law,n", [("grav", 1001), ("grav", 4001), ("grav", 5001), ("grav", 12289),
                                   ("ljc", 777), ("ljc", 2433), ("ljc", 8192)])
def test_steps(law, n):
    nb = lib()
    pos, vel, prm, kw = _system(law, n)
    acc = _shifted(nb.forces(pos, prm, **kw))
    outs = []
    for split in (1, 8):
        p, v, a = (_shifted(t) for t in (pos, vel, acc))
        for _ in range(split):
            nb.step(p, v, a, prm, dt=1e-4, nsteps=8 // split, acc_valid=True, **kw)
        outs.append((p, v, a))
    _same(outs)


@pytest.mark.parametrize("n", [1001, 2433, 8191])
def test_hermite(n):
    nb = lib()
    pos, vel, _, kw = _system("grav", n)
    outs = []
    for split in (1, 6):
        p, v = _shifted(pos), _shifted(vel)
        a, j = _shifted(pos), _shifted(pos)
        for k in range(split):
            nb.hermite_step(p, v, a, j, dt=1e-4, nsteps=6 // split, acc_valid=k > 0, **kw)
        outs.append((p, v, a, j))
    _same(outs)


@pytest.mark.parametrize("law,n", [("grav", 1001), ("grav", 2433), ("grav", 8191), ("ljc", 777),
                                   ("ljc", 2561)])
def test_reverse_sweep(law, n):
    nb = lib()
    pos, vel, prm, kw = _system(law, n)
    k = 5
    xs = torch.cat([pos + 1e-3 * s * vel for s in range(k)])
    lam = np.random.default_rng(n).standard_normal((2, n, 4)).astype(np.float32)
    lam[:, :, 3] = 0.0
    outs = []
    for split in (1, k):
        lx, lv = (_shifted(torch.from_numpy(t).to(dev())) for t in lam)
        gm = torch.zeros(n, device=dev())
        gt = torch.zeros(8, dtype=torch.float64, device=dev())
        m = k // split
        for c in range(split - 1, -1, -1):
            nb.api.adjoint_leapfrog(_shifted(xs[c * m * n:(c + 1) * m * n]), lx, lv, prm, k=m,
                                    dt=1e-3, first=False, grad_m=gm,
                                    grad_types=None if prm is None else gt, **kw)
        outs.append((lx, lv, gm))
    _same(outs)


def test_batch():
    nb = lib()
    table, at, parts = [], 0, []
    for k, n in enumerate((2305, 700, 1501, 64, 900)):
        pos, vel = grav_tensors(workloads.plummer(n, seed=n, eps=0.01))
        table.append(dict(offset=at, n=n, law=nb.LAW_GRAV, eps=0.01, dt=1e-3))
        parts.append((pos, vel))
        at += n
    pos, vel = (torch.cat([p[c] for p in parts]) for c in (0, 1))
    plan = nb.BatchPlan(table)
    acc = torch.zeros_like(pos)
    plan.run(pos, vel, acc, nsteps=0, graph=False)
    outs = []
    for split in (1, 6):
        p, v, a = _shifted(pos), _shifted(vel), _shifted(acc)
        for _ in range(split):
            plan.run(p, v, a, nsteps=6 // split, acc_valid=True, graph=False)
        outs.append((p, v, a))
    _same(outs)
