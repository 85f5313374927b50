"""GPU parity of the batched streamed triangle kernel that default plans run: systems at
the edges of its rows (384 targets for gravity, 256 for the LJC laws) and source groups
(32), cut into one and into several segments, with unused particles between the systems,
against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_util import assert_forces_close, dev, lib

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 32, 33, 255, 256, 257, 383, 384, 385, 769, 1100]


def _table(sizes, gap=2):
    nb = lib()
    laws = (nb.LAW_GRAV, nb.LAW_LJC, nb.LAW_LJC_LINEAR)
    total = sum(3 * (n + gap) for n in sizes)
    pos = np.zeros((total, 4), np.float32)
    pos[:, 3] = 1.0
    vel = np.zeros((total, 4), np.float32)
    q, sg, ep = np.zeros(total), np.full(total, 3.0), np.full(total, 0.1)
    ty = np.zeros(total, np.int32)
    used = np.zeros(total, bool)
    table, refs, at = [], [], 0
    for n in sizes:
        for law in laws:
            if law == nb.LAW_GRAV:
                s = workloads.plummer(n, seed=n, eps=0.01)
                x, v, m = s.f32()
                eps = float(np.float32(s.eps))
                xd, _, md = s.f32_as_f64()
                refs.append(oracle.GravSystem(md, eps=eps).accel(xd) if n > 1 else None)
                table.append(dict(offset=at, n=n, law=law, G=1.0, eps=eps, dt=1e-3))
            else:
                s = workloads.ljc_sphere(n, seed=n)
                x, v, m, qq, st, et = s.f32()
                xd, _, md, qd, sd, ed = s.f32_as_f64()
                lin = law == nb.LAW_LJC_LINEAR
                refs.append(oracle.LJCSystem(md, qd, s.types, sd, ed, 332.0637 / 80.0,
                                             linear=lin).accel(xd) if n > 1 else None)
                i = slice(at, at + n)
                q[i], sg[i], ep[i], ty[i] = qd, sd[s.types], ed[s.types], s.types
                table.append(dict(offset=at, n=n, law=law, dt=1e-5))
            pos[at:at + n, :3], pos[at:at + n, 3], vel[at:at + n, :3] = x, m, v
            used[at:at + n] = True
            at += n + gap
    d = dev()
    prm = nb.pack_ljc(*(torch.from_numpy(a).to(d) for a in (q, sg, ep, ty)), kq=332.0637 / 80.0)
    return torch.from_numpy(pos).to(d), torch.from_numpy(vel).to(d), prm, table, refs, used


@pytest.mark.parametrize("mode", ["plain", "precise", "uncompensated"])
@pytest.mark.parametrize("sizes", [SIZES, [4100, 40, 2304], [64] * 40])
def test_forces_and_steps(mode, sizes):
    nb = lib()
    pos, vel, prm, table, refs, used = _table(sizes)
    plan = nb.BatchPlan(table, precise=mode == "precise", compensated=mode != "uncompensated")
    acc = torch.full_like(pos, 7.0)
    plan.run(pos, vel, acc, prm, nsteps=0, graph=False)
    a = acc.cpu().numpy()
    for s, ref in zip(table, refs):
        got = a[s["offset"]:s["offset"] + s["n"], :3]
        if ref is None:
            assert not got.any()
        else:
            assert_forces_close(got, ref, what=f"law {s['law']} n={s['n']}")
    assert (a[~used] == 7.0).all()  # particles of no system are left alone
    # steps, captured and eager, in one call and one by one
    outs = []
    for graph, split in ((True, 1), (False, 1), (False, 4)):
        p, v, b = pos.clone(), vel.clone(), acc.clone()
        for k in range(split):
            plan.run(p, v, b, prm, nsteps=4 // split, acc_valid=True, graph=graph)
        torch.cuda.synchronize()
        outs.append((p, v, b))
    for other in outs[1:]:
        for s, t in zip(outs[0], other):
            assert torch.equal(s, t)
    assert torch.equal(outs[0][0][~torch.from_numpy(used).to(dev())],
                       pos[~torch.from_numpy(used).to(dev())])
    nb.sync_check()
