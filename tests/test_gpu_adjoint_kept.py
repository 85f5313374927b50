"""Reverse leapfrog with all positions kept, with only the newest chunks' kept and the
others recomputed from checkpoints, and with a chunk length that does not divide the
steps: the same gradients bit for bit."""
import numpy as np
import pytest
import torch

import workloads
from gpu_util import dev, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("law", ["grav", "ljc"])
@pytest.mark.parametrize("n", [300, 2600])
def test_kept_and_recomputed_positions(law, n, monkeypatch):
    nb = lib()
    from paper_0706_3060_gb300 import autograd
    d = dev()
    if law == "grav":
        g = workloads.plummer(n, seed=n, eps=0.01)
        x, v, m = g.f32()
        kw, extra = dict(eps=float(np.float32(g.eps)), dt=1e-3), ()
    else:
        s = workloads.ljc_sphere(n, seed=n)
        x, v, m, q, st, et = s.f32()
        kw = dict(law=nb.LAW_LJC, dt=1e-5, q=torch.from_numpy(q.astype(np.float64)).to(d),
                  types=torch.from_numpy(s.types).to(d))
        extra = tuple(torch.from_numpy(a).to(d).requires_grad_(True) for a in (st, et))
        kw.update(sig_t=extra[0], eps_t=extra[1])
    w = torch.from_numpy(np.random.default_rng(3).standard_normal((2, n, 3))
                         .astype(np.float32)).to(d)

    def grads(k, kept):
        if kept is not None:
            monkeypatch.setattr(autograd, "_kept_steps", lambda *a: kept)
        leaves = [torch.from_numpy(np.ascontiguousarray(a)).to(d).requires_grad_(True)
                  for a in (x, v, m)]
        xT, vT = autograd.leapfrog(*leaves, nsteps=7, k=k, **kw)
        out = torch.autograd.grad([xT, vT], leaves + list(extra), [w[0], w[1]])
        monkeypatch.undo()
        return out

    base = grads(2, None)
    for k, kept in ((2, 2), (2, 4), (3, 3), (3, 100), (7, 7)):
        got = grads(k, kept)
        for a, b in zip(base[:3], got[:3]):
            assert torch.equal(a, b), (k, kept)
        for a, b in zip(base[3:], got[3:]):  # per-type sums: a different order of additions
            torch.testing.assert_close(a, b, rtol=1e-6, atol=0)
    nb.sync_check()
