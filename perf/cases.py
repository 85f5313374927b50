"""Performance cases of the all-pairs N-body library: calls that a simulation program
makes through the package's public functions, over the sizes it makes them at.

A case is a dict of plain values. ``kind`` names the call:

* ``forces``  -- one force evaluation (gravity, or LJ + Coulomb with a constant or a
  linear dielectric), optionally with the potential;
* ``steps``   -- leapfrog steps from a carried acceleration, optionally with the
  two-float state;
* ``hermite`` -- fourth-order Hermite steps on acceleration and jerk;
* ``subset``  -- forces on a list of active particles against all (block time steps);
* ``batch``   -- leapfrog steps of an ensemble of small systems of both laws;
* ``grad``    -- a differentiable run of leapfrog steps and its backward pass.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_0706_3060_gb300 as nb
from paper_0706_3060_gb300.autograd import leapfrog

DEV = "cuda"
LAWS = {"grav": nb.LAW_GRAV, "ljc": nb.LAW_LJC, "ljclin": nb.LAW_LJC_LINEAR}
# Coulomb prefactor: k_e / 80 (constant) and k_e / (4 r) (linear dielectric).
KQ = {"ljc": nb.COULOMB_K / 80.0, "ljclin": nb.COULOMB_K / 4.0}
ATOM_MASSES = (12.011, 14.007, 15.999, 32.06)
SIG_T = (2.6, 2.9, 3.3, 3.7)  # Angstrom, per type
EPS_T = (0.06, 0.1, 0.14, 0.19)  # kcal/mol, per type


def listed():
    return [
        # A cluster small enough that a program waits on launches rather than on arithmetic:
        # the small gravity workload, called once per step by an integrator of the user's own.
        dict(name="forces_1024", kind="forces", law="grav", n=1024, pot=False),
        # A small solvated protein, 1280 atoms: one energy and force evaluation of a minimizer.
        dict(name="forces_ljc_1280", kind="forces", law="ljc", n=1280, pot=True),
        # A star cluster of a few thousand members (an odd count) followed for some steps.
        dict(name="steps_4001", kind="steps", law="grav", n=4001, nsteps=20, two=False),
        # Molecular dynamics of the 8192-atom sphere.
        dict(name="steps_ljc_8192", kind="steps", law="ljc", n=8192, nsteps=10, two=False),
        # One step of the large gravity workload.
        dict(name="step_262144", kind="steps", law="grav", n=262144, nsteps=1, two=False),
        # Forces and potential of a mid-size galaxy model, with a count that fits no tile.
        dict(name="forces_pot_50021", kind="forces", law="grav", n=50021, pot=True),
        # A large molecule with the linear dielectric, at an odd atom count.
        dict(name="forces_ljclin_30011", kind="forces", law="ljclin", n=30011, pot=False),
        # Collisional dynamics with the Hermite scheme.
        dict(name="hermite_32768", kind="hermite", law="grav", n=32768, nsteps=2),
        # One rung of a block time-step scheme: a few percent of the particles are due.
        dict(name="subset_65536", kind="subset", law="grav", n=65536, active=1500),
        # Many small systems of uneven size advanced together.
        dict(name="batch_512", kind="batch", law="mixed", n=4096, nsys=512, nsteps=5),
        # Gradients through a gravity run (initial conditions fitted to a target).
        dict(name="grad_16384", kind="grad", law="grav", n=16384, nsteps=40, k=10),
        # Gradients of a molecular run with respect to its atom parameters.
        dict(name="grad_ljc_8192", kind="grad", law="ljc", n=8192, nsteps=10, k=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(["forces", "forces", "steps", "steps", "hermite", "subset", "batch",
                           "grad"])
        law = rng.choice(["grav", "grav", "ljc", "ljclin"])
        if kind in ("hermite", "subset"):
            law = "grav" if kind == "hermite" else law
        if kind == "forces":
            c = dict(kind=kind, law=law, n=_log_int(rng, 256, 262144 if law == "grav" else 65536),
                     pot=rng.random() < 0.5)
        elif kind == "steps":
            c = dict(kind=kind, law=law, n=_log_int(rng, 1000, 262144 if law == "grav" else 65536),
                     nsteps=_log_int(rng, 1, 40), two=rng.random() < 0.3)
        elif kind == "hermite":
            c = dict(kind=kind, law=law, n=_log_int(rng, 1000, 131072),
                     nsteps=_log_int(rng, 1, 20))
        elif kind == "subset":
            n = _log_int(rng, 4096, 131072)
            c = dict(kind=kind, law=law, n=n, active=_log_int(rng, 32, n // 8))
        elif kind == "batch":
            c = dict(kind=kind, law="mixed", n=_log_int(rng, 512, 4096),
                     nsys=_log_int(rng, 16, 512), nsteps=_log_int(rng, 1, 10))
        else:
            nsteps = _log_int(rng, 4, 40)
            c = dict(kind=kind, law=law, n=_log_int(rng, 1000, 20000), nsteps=nsteps,
                     k=rng.randint(2, nsteps))
        if work(c)["flops"] <= most:
            return c


# ---- inputs ------------------------------------------------------------------------------
def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _softening(n):
    return float(np.float32(0.01 if n < 16384 else 0.04 * n ** (-1.0 / 3.0)))


def _sphere_dirs(rng, n):
    u = rng.uniform(-1.0, 1.0, n)
    p = rng.uniform(0.0, 2.0 * math.pi, n)
    s = np.sqrt(1.0 - u * u)
    return np.stack([s * np.cos(p), s * np.sin(p), u], 1)


def _cluster(rng, n):
    """Plummer sphere in virial units (G = M = a = 1) with unequal masses:
    FP32 (n, 4) positions with masses, and velocities."""
    r = 1.0 / np.sqrt(rng.uniform(1e-9, 0.999, n) ** (-2.0 / 3.0) - 1.0)
    x = r[:, None] * _sphere_dirs(rng, n)
    q = np.empty(n)
    todo = np.arange(n)
    while todo.size:  # speeds by rejection from q^2 (1 - q^2)^(7/2)
        a, b = rng.uniform(0.0, 1.0, (2, todo.size))
        ok = 0.1 * b < a * a * (1.0 - a * a) ** 3.5
        q[todo[ok]] = a[ok]
        todo = todo[~ok]
    v = (q * math.sqrt(2.0) * (1.0 + r * r) ** -0.25)[:, None] * _sphere_dirs(rng, n)
    m = rng.uniform(0.5, 1.5, n)
    m /= m.sum()
    x -= (m[:, None] * x).sum(0)
    v -= (m[:, None] * v).sum(0)
    return _f4(x, m), _f4(v, np.zeros(n))


def _molecule(rng, n):
    """Atoms at liquid density (46.6 A^3 each, as in a 45 A sphere of 8192): a jittered
    lattice cut to a ball, in random order, with thermal velocities. Returns positions with
    masses, velocities, charges and types."""
    a = 3.6
    h = int(math.ceil((3.0 * n / (4.0 * math.pi)) ** (1.0 / 3.0))) + 2
    ax = np.arange(-h, h + 1) * a
    g = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    g = g + rng.uniform(-0.5 * a, 0.5 * a, 3)
    g = g[np.argsort((g * g).sum(1), kind="stable")[:n]]
    x = g[rng.permutation(n)] + rng.uniform(-0.3, 0.3, (n, 3))
    types = rng.integers(0, 4, n).astype(np.int32)
    m = np.asarray(ATOM_MASSES)[types]
    v = rng.standard_normal((n, 3)) * np.sqrt(0.593 / m)[:, None]
    q = rng.uniform(-0.8, 0.8, n).astype(np.float32).astype(np.float64)
    return _f4(x, m), _f4(v, np.zeros(n)), q, types


def _f4(x, w):
    return np.concatenate([x, np.asarray(w)[:, None]], 1).astype(np.float32)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _prm(q, types, law):
    t = torch.from_numpy(types).to(DEV)
    sig = torch.tensor(SIG_T, dtype=torch.float32).double().to(DEV)[t.long()]
    eps = torch.tensor(EPS_T, dtype=torch.float32).double().to(DEV)[t.long()]
    return nb.pack_ljc(_gpu(q), sig, eps, t, kq=KQ[law])


def _single(case, seed):
    """Host arrays of a one-system case: pos, vel, charges, types."""
    rng = _rng(seed)
    if case["law"] == "grav":
        return _cluster(rng, case["n"]) + (None, None)
    return _molecule(rng, case["n"])


def _dt(law):
    return 1e-4 if law == "grav" else 1e-2


def _ensemble(case, seed):
    """Systems of log-uniform size between 64 and case["n"], gravity and LJ + Coulomb in
    turn: the table, pos, vel, charges and types of all, back to back."""
    rng = _rng(seed)
    sizes = _rng(7).uniform(math.log(64), math.log(case["n"]), case["nsys"])
    table, pos, vel, q, types, off = [], [], [], [], [], 0
    for k, s in enumerate(sizes):
        n = int(round(math.exp(s)))
        if k % 2 == 0:
            p, v = _cluster(rng, n)
            qq, tt = np.zeros(n), np.zeros(n, np.int32)
            table.append(dict(offset=off, n=n, law=nb.LAW_GRAV, eps=_softening(n), dt=1e-3))
        else:
            p, v, qq, tt = _molecule(rng, n)
            table.append(dict(offset=off, n=n, law=nb.LAW_LJC, dt=1e-2))
        pad = -n % 4  # offsets are multiples of 4
        for lst, a in ((pos, p), (vel, v), (q, qq), (types, tt)):
            lst.append(np.concatenate([a, np.zeros((pad,) + a.shape[1:], a.dtype)]))
        off += n + pad
    return (table,) + tuple(np.concatenate(a) for a in (pos, vel, q, types))


def prepare(case, seed):
    kind, law, n = case["kind"], case["law"], case["n"]
    st = dict(case=case, law=LAWS.get(law))
    if kind == "batch":
        table, pos, vel, q, types = _ensemble(case, seed)
        st.update(pos=_gpu(pos), vel=_gpu(vel), prm=_prm(q, types, "ljc"))
        st["plan"] = nb.BatchPlan(table)
        st["acc"] = torch.zeros_like(st["pos"])
        st["plan"].run(st["pos"], st["vel"], st["acc"], st["prm"], nsteps=0, graph=False)
        return st
    pos, vel, q, types = _single(case, seed)
    st["eps"] = _softening(n) if law == "grav" else 0.0
    st["pos"], st["vel"] = _gpu(pos), _gpu(vel)
    st["prm"] = None if law == "grav" else _prm(q, types, law)
    if kind == "steps":
        st["acc"] = nb.forces(st["pos"], st["prm"], law=st["law"], eps=st["eps"])
        if case["two"]:
            st["lo"] = torch.zeros((2 * n, 4), dtype=torch.float32, device=DEV)
    elif kind == "hermite":
        st["acc"], st["jerk"] = nb.forces_jerk(st["pos"], st["vel"], eps=st["eps"])
    elif kind == "subset":
        st["idx"] = _gpu(_rng(seed + 1).permutation(n)[:case["active"]].astype(np.int32))
    elif kind == "grad":
        st["leaves"] = [st["pos"][:, :3].clone().requires_grad_(True),
                        st["vel"][:, :3].clone().requires_grad_(True),
                        st["pos"][:, 3].clone().requires_grad_(True)]
        gx, gv = _cotangents(case, seed)
        st["gx"], st["gv"] = gx.float(), gv.float()
        if law != "grav":
            st["leaves"] += [torch.tensor(SIG_T, device=DEV).requires_grad_(True),
                             torch.tensor(EPS_T, device=DEV).requires_grad_(True)]
            st["ff"] = dict(q=_gpu(q), types=_gpu(types), kq=KQ[law])
    return st


def _cotangents(case, seed):
    """dL/dx_T and dL/dv_T, as FP64 tensors holding FP32 values."""
    rng = _rng(seed + 2)
    g = rng.standard_normal((2, case["n"], 3)).astype(np.float32)
    return _gpu(g[0]).double(), _gpu(g[1]).double()


def run(state):
    c = state["case"]
    kind = c["kind"]
    pos, vel, law = state["pos"], state["vel"], state["law"]
    if kind == "forces":
        return nb.forces(pos, state["prm"], law=law, eps=state["eps"], pot=c["pot"])
    if kind == "steps":
        nb.step(pos, vel, state["acc"], state["prm"], dt=_dt(c["law"]), nsteps=c["nsteps"],
                law=law, eps=state["eps"], acc_valid=True, state_lo=state.get("lo"))
        return pos, vel, state["acc"]
    if kind == "hermite":
        nb.hermite_step(pos, vel, state["acc"], state["jerk"], dt=1e-4, nsteps=c["nsteps"],
                        eps=state["eps"], acc_valid=True)
        return pos, vel, state["acc"], state["jerk"]
    if kind == "subset":
        return nb.forces_subset(pos, state["idx"], state["prm"], law=law, eps=state["eps"])
    if kind == "batch":
        state["plan"].run(pos, vel, state["acc"], state["prm"], nsteps=c["nsteps"],
                          acc_valid=True)
        return pos, vel, state["acc"]
    x0, v0, m = state["leaves"][:3]
    more = dict(state["ff"], sig_t=state["leaves"][3], eps_t=state["leaves"][4]) \
        if "ff" in state else {}
    xT, vT = leapfrog(x0, v0, m, dt=_dt(c["law"]), nsteps=c["nsteps"], k=c["k"],
                      eps=state["eps"], law=law, **more)
    grads = torch.autograd.grad([xT, vT], state["leaves"], [state["gx"], state["gv"]])
    return (xT.detach(), vT.detach()) + tuple(grads)


# ---- the least work of a pass ----------------------------------------------------------------
# FP32 operations of one unordered pair applied to both particles (a fused multiply-add is two).
PAIR_FLOPS = {"grav": 26, "ljc": 37, "ljclin": 38}
POT_FLOPS = {"grav": 4, "ljc": 7, "ljclin": 7}
VJP_FLOPS = {"grav": 58, "ljc": 95, "ljclin": 96}


def work(case):
    kind, law, n = case["kind"], case["law"], case["n"]
    pairs = 0.5 * n * (n - 1)
    f4 = 16 * n
    prm = 0 if law == "grav" else f4
    if kind == "forces":
        f = PAIR_FLOPS[law] + (POT_FLOPS[law] if case["pot"] else 0)
        return dict(bytes=2 * f4 + prm, flops=f * pairs)
    if kind == "steps":
        return dict(bytes=(10 if case["two"] else 6) * f4 + prm,
                    flops=PAIR_FLOPS[law] * pairs * case["nsteps"])
    if kind == "hermite":
        return dict(bytes=8 * f4, flops=51 * pairs * case["nsteps"])
    if kind == "subset":  # ordered pairs: one side only
        a = case["active"]
        return dict(bytes=f4 + prm + 20 * a, flops=(PAIR_FLOPS[law] - 7) * float(a) * n)
    if kind == "batch":
        sizes = np.rint(np.exp(_rng(7).uniform(math.log(64), math.log(n), case["nsys"])))
        fl = sum(0.5 * s * (s - 1) * PAIR_FLOPS["ljc" if k % 2 else "grav"]
                 for k, s in enumerate(sizes))
        return dict(bytes=float(7 * 16 * sizes.sum()), flops=float(fl) * case["nsteps"])
    t = case["nsteps"]  # forward evaluations, then one product per step and the final kick's
    return dict(bytes=12 * f4 + prm,
                flops=pairs * (PAIR_FLOPS[law] * (t + 1) + VJP_FLOPS[law] * (t + 1)))


# ---- 64-bit values -------------------------------------------------------------------------
def _accel64(x, m, law, eps2, q=None, sig=None, eps=None, rows=None, want_pot=False, mrow=None):
    """Accelerations (and potentials) of the particles `rows` (a slice or an index tensor)
    by direct sums in 64 bits. law: grav, ljc or ljclin; q already scaled by sqrt(kq)."""
    xi = x[rows]
    d = x[None, :, :] - xi[:, None, :]
    r2 = (d * d).sum(-1) + (eps2 if law == "grav" else 0.0)
    idx = torch.arange(x.shape[0], device=x.device)
    self_pair = idx[None, :] == idx[rows][:, None]
    y = torch.where(self_pair, torch.zeros_like(r2),
                    torch.where(self_pair, torch.ones_like(r2), r2).rsqrt())
    if law == "grav":
        a = (m[None, :, None] * (y * y * y)[..., None] * d).sum(1)
        return a, (-(m[None, :] * y).sum(1) if want_pot else None)
    y2 = y * y
    qq = q[rows][:, None] * q[None, :]
    s = 0.5 * (sig[rows][:, None] + sig[None, :])
    e = 4.0 * (eps[rows][:, None] * eps[None, :]).sqrt()
    u = (s * s * y2) ** 3
    coul = qq * y * y2 if law == "ljc" else 2.0 * qq * y2 * y2
    f = coul + 6.0 * e * y2 * (2.0 * u * u - u)
    a = -(f[..., None] * d).sum(1) / m[rows][:, None]
    if not want_pot:
        return a, None
    return a, (qq * (y if law == "ljc" else y2) + e * (u * u - u)).sum(1)


def _all64(x, m, law, eps2, ff=(), want_pot=False):
    n = x.shape[0]
    ch = max(1, (1 << 25) // n)
    out = [_accel64(x, m, law, eps2, *ff, rows=slice(b, min(b + ch, n)), want_pot=want_pot)
           for b in range(0, n, ch)]
    return torch.cat([o[0] for o in out]), torch.cat([o[1] for o in out]) if want_pot else None


def _ff64(q, types, law):
    t = torch.from_numpy(types).long().to(DEV)
    sig = torch.tensor(SIG_T, dtype=torch.float32).double().to(DEV)
    eps = torch.tensor(EPS_T, dtype=torch.float32).double().to(DEV)
    return _gpu(q) * math.sqrt(KQ[law]), t, sig, eps


def _w4(xyz, w=None):
    w = torch.zeros_like(xyz[:, 0]) if w is None else w
    return torch.cat([xyz, w[:, None]], 1)


def _leap64(x, v, acc, dt, nsteps):
    """Kick-drift-kick; returns x, v, a and the positions before each drift."""
    a, xs = acc(x), []
    for _ in range(nsteps):
        xs.append(x)
        v = v + 0.5 * dt * a
        x = x + dt * v
        a = acc(x)
        v = v + 0.5 * dt * a
    return x, v, a, xs


def exact(case, seed):
    kind, law, n = case["kind"], case["law"], case["n"]
    if kind == "batch":
        return _exact_batch(case, seed)
    pos, vel, q, types = _single(case, seed)
    p, v = _gpu(pos).double(), _gpu(vel).double()[:, :3]
    x, m = p[:, :3].contiguous(), p[:, 3].contiguous()
    eps2 = float(np.float32(_softening(n) ** 2)) if law == "grav" else 0.0
    ff, sig_t, eps_t, t = (), None, None, None
    if law != "grav":
        qs, t, sig_t, eps_t = _ff64(q, types, law)
        ff = (qs, sig_t[t], eps_t[t])
    if kind == "forces":
        a, phi = _all64(x, m, law, eps2, ff, want_pot=case["pot"])
        return _w4(a, phi)
    if kind == "subset":
        idx = _gpu(_rng(seed + 1).permutation(n)[:case["active"]])
        ch = max(1, (1 << 25) // n)
        a = [_accel64(x, m, law, eps2, *ff, rows=idx[b:b + ch])[0]
             for b in range(0, len(idx), ch)]
        return _w4(torch.cat(a))
    if kind == "steps":
        dt = float(np.float32(_dt(law)))
        x, v, a, _ = _leap64(x, v, lambda y: _all64(y, m, law, eps2, ff)[0], dt, case["nsteps"])
        return _w4(x, m), _w4(v), _w4(a)
    if kind == "hermite":
        return _exact_hermite(case, x, v, m, eps2)
    return _exact_grad(case, seed, x, v, m, eps2, ff, sig_t, eps_t, t)


def _jerk64(x, v, m, eps2):
    n = x.shape[0]
    ch = max(1, (1 << 24) // n)
    out = []
    for b in range(0, n, ch):
        d = x[None] - x[b:b + ch, None]
        u = v[None] - v[b:b + ch, None]
        y2 = 1.0 / ((d * d).sum(-1) + eps2)
        w = (m[None] * y2 * y2.sqrt())[..., None]
        c = -3.0 * y2 * (d * u).sum(-1)
        out.append(((w * d).sum(1), (w * (u + c[..., None] * d)).sum(1)))
    return torch.cat([o[0] for o in out]), torch.cat([o[1] for o in out])


def _exact_hermite(case, x, v, m, eps2):
    dt = float(np.float32(1e-4))
    a, j = _jerk64(x, v, m, eps2)
    for _ in range(case["nsteps"]):
        xp = x + dt * v + dt * dt / 2 * a + dt ** 3 / 6 * j
        vp = v + dt * a + dt * dt / 2 * j
        a1, j1 = _jerk64(xp, vp, m, eps2)
        v1 = v + dt / 2 * (a + a1) + dt * dt / 12 * (j - j1)
        x = x + dt / 2 * (v + v1) + dt * dt / 12 * (a - a1)
        v, a, j = v1, a1, j1
    return _w4(x, m), _w4(v), _w4(a), _w4(j)


def _exact_grad(case, seed, x, v, m, eps2, ff, sig_t, eps_t, t):
    law, n, steps = case["law"], case["n"], case["nsteps"]
    dt = float(np.float32(_dt(law)))
    xT, vT, _, xs = _leap64(x, v, lambda y: _all64(y, m, law, eps2, ff)[0], dt, steps)
    lx, lv = _cotangents(case, seed)
    grads = [torch.zeros_like(m)] + ([] if t is None else [torch.zeros_like(sig_t),
                                                          torch.zeros_like(eps_t)])
    ch = max(1, (1 << 23) // n)

    def pull(at, lam, w):
        """Adds w J^T lam of the accelerations at `at` to the parameters' gradients and
        returns its position part."""
        ins = [at.clone().requires_grad_(True), m.clone().requires_grad_(True)]
        if t is not None:
            ins += [sig_t.clone().requires_grad_(True), eps_t.clone().requires_grad_(True)]
        gx = torch.zeros_like(at)
        for b in range(0, n, ch):
            sub = slice(b, min(b + ch, n))
            f = () if t is None else (ff[0], ins[2][t], ins[3][t])
            with torch.enable_grad():
                a, _ = _accel64(ins[0], ins[1], law, eps2, *f, rows=sub)
                got = torch.autograd.grad((a * lam[sub]).sum(), ins)
            gx += w * got[0]
            for k in range(1, len(ins)):
                grads[k - 1] += w * got[k]
        return gx

    lx = lx + pull(xT, lv, 0.5 * dt)
    for s in range(steps - 1, -1, -1):
        lv = lv + dt * lx
        lx = lx + pull(xs[s], lv, 0.5 * dt if s == 0 else dt)
    return (xT, vT, lx, lv) + tuple(grads)


def _exact_batch(case, seed):
    table, pos, vel, q, types = _ensemble(case, seed)
    out = [_gpu(pos).double(), _gpu(vel).double(), torch.zeros(pos.shape, device=DEV).double()]
    for s in table:
        sl = slice(s["offset"], s["offset"] + s["n"])
        x, v, m = out[0][sl, :3].clone(), out[1][sl, :3].clone(), out[0][sl, 3].clone()
        grav = s["law"] == nb.LAW_GRAV
        ff = ()
        if not grav:
            qs, t, sig_t, eps_t = _ff64(q[sl], types[sl], "ljc")
            ff = (qs, sig_t[t], eps_t[t])
        eps2 = float(np.float32(s["eps"] ** 2)) if grav else 0.0
        law = "grav" if grav else "ljc"
        x, v, a, _ = _leap64(x, v, lambda y: _all64(y, m, law, eps2, ff)[0],
                             float(np.float32(s["dt"])), case["nsteps"])
        out[0][sl], out[1][sl], out[2][sl] = _w4(x, m), _w4(v), _w4(a)
    return tuple(out)
