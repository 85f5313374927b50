"""Reverse-mode leapfrog as a torch.autograd.Function with checkpointing.

Forward: ``nsteps`` KDK steps through nbody_step with the compensated two-float
state, in chunks of ``k`` steps. The positions of the newest chunks are stored, as
many as fit the budget of :func:`_kept_steps`; of an older chunk only the state at
its start (x, v, low parts and a), a checkpoint. Backward: for each chunk, newest
first, run the reverse sweep nbody_adjoint_leapfrog (force VJP kernels + fused
adjoint updates) over the chunk's positions; those of a checkpointed chunk are
recomputed with nbody_step's trace on a second stream while the sweep of the
next-newer chunk runs, so the two fill each other's partial waves: k - 1 force
evaluations per chunk of k steps.
With merged half-kicks the sweep is

    lam_x += dt/2 J(x_T)^T lam_v                      (only if dL/dv_T != 0)
    for n = T-1 .. 0:  lam_v += dt lam_x;  lam_x += w_n J(x_n)^T lam_v
                       (w_n = dt, w_0 = dt/2)

and returns dL/dx_0 = lam_x, dL/dv_0 = lam_v, dL/dm and, for LJC, dL/dsigma_t
and dL/deps_t. All arithmetic runs in the library's kernels.
"""
from __future__ import annotations

import torch

from . import api
from ._lib import LAW_GRAV, LAW_LJC, LAW_LJC_LINEAR

_LJC_LAWS = (LAW_LJC, LAW_LJC_LINEAR)

_SIDE: dict = {}  # device index -> the stream that recomputes chunk positions


def _side_stream(dev):
    idx = dev.index if dev.index is not None else torch.cuda.current_device()
    if idx not in _SIDE:
        _SIDE[idx] = torch.cuda.Stream(device=dev)
    return _SIDE[idx]


class _Cfg:
    def __init__(self, law, dt, nsteps, k, G, eps, q=None, types=None, kq=None, ntypes=4,
                 keep_bytes=None):
        self.law, self.dt, self.nsteps, self.k = law, float(dt), int(nsteps), int(k)
        self.keep_bytes = keep_bytes
        self.G, self.eps = float(G), float(eps)
        self.q, self.types, self.kq, self.ntypes = q, types, kq, ntypes


_KEEP_ALWAYS = 32 << 20  # bytes of positions that are kept without asking what is free


def _kept_steps(n, nsteps, k, dev, keep_bytes=None):
    """Steps, counted from the last, whose positions the forward pass keeps (16 bytes a
    particle and step, and once more per chunk). All of them where they take no more than
    the checkpoints would (80 bytes a particle and chunk, and the newest chunk's positions);
    else as many as fit in ``keep_bytes``, or without it in 32 MiB, or in a 256th of the
    device's memory and a 64th of what is free of it, so that several graphs alive at once
    leave each other room; always the newest chunk's. Each step kept is a force evaluation
    that the backward pass need not repeat (40 steps of 16384 particles, k = 10: 27 of 108
    evaluations and products, 12.6 ms -> 10.3)."""
    row = 16 * max(n, 1)
    chunks = -(-nsteps // k)
    if nsteps + chunks <= 5 * chunks + k:
        return nsteps
    if keep_bytes is None:
        keep_bytes = _KEEP_ALWAYS
        if row * (nsteps + chunks) > keep_bytes and not torch.cuda.is_current_stream_capturing():
            free, total = torch.cuda.mem_get_info(dev)
            free += torch.cuda.memory_reserved(dev) - torch.cuda.memory_allocated(dev)
            keep_bytes = max(keep_bytes, min(total // 256, free // 64))
    return max(k, keep_bytes // row * k // (k + 1))


def _prm(cfg, sig_t, eps_t):
    if cfg.law not in _LJC_LAWS:
        return None
    t = cfg.types.long()
    return api.pack_ljc(cfg.q, sig_t.double()[t], eps_t.double()[t], cfg.types, kq=cfg.kq)


class NBodyLeapfrog(torch.autograd.Function):
    """(x0, v0, m, sig_t, eps_t) -> (x_T, v_T) through ``nsteps`` leapfrog steps."""

    @staticmethod
    def forward(ctx, x0, v0, m, sig_t, eps_t, cfg):
        dev = x0.device
        n = x0.shape[0]
        pos = torch.empty((n, 4), dtype=torch.float32, device=dev)
        pos[:, :3] = x0.detach()
        pos[:, 3] = m.detach()
        vel = torch.zeros((n, 4), dtype=torch.float32, device=dev)
        vel[:, :3] = v0.detach()
        acc = torch.empty_like(pos)
        lo = torch.zeros((2 * n, 4), dtype=torch.float32, device=dev)  # two-float state
        prm = _prm(cfg, sig_t, eps_t)
        chunks = []  # (positions, None) or (None, checkpoint) of each chunk
        done = 0
        kept = _kept_steps(n, cfg.nsteps, cfg.k, dev, cfg.keep_bytes)
        while done < cfg.nsteps:
            steps = min(cfg.k, cfg.nsteps - done)
            trace = ckpt = None
            if cfg.nsteps - done <= kept:
                trace = torch.empty(((steps + 1) * n, 4), dtype=torch.float32, device=dev)
            else:
                # the checkpoint keeps a(x) at its positions too (carried in from the
                # previous chunk), so that its recompute starts without an evaluation
                ckpt = (pos.clone(), vel.clone(), lo.clone(), acc.clone() if done > 0 else None)
            chunks.append((trace, ckpt))
            api.step(pos, vel, acc, prm, dt=cfg.dt, nsteps=steps, law=cfg.law, G=cfg.G,
                     eps=cfg.eps, acc_valid=done > 0, state_lo=lo, trace=trace)
            done += steps
        ctx.cfg = cfg
        ctx.chunks = chunks
        ctx.prm = prm
        ctx.save_for_backward(pos)
        return pos[:, :3].clone(), vel[:, :3].clone()

    @staticmethod
    def backward(ctx, gx, gv):
        cfg = ctx.cfg
        (pos_T,) = ctx.saved_tensors
        n = pos_T.shape[0]
        dev = pos_T.device
        lam_x = torch.zeros((n, 4), dtype=torch.float32, device=dev)
        lam_v = torch.zeros((n, 4), dtype=torch.float32, device=dev)
        if gx is not None:
            lam_x[:, :3] = gx
        if gv is not None:
            lam_v[:, :3] = gv
        grad_m = torch.zeros(n, dtype=torch.float32, device=dev)
        grad_t = torch.zeros(2 * cfg.ntypes, dtype=torch.float64, device=dev)
        gt = grad_t if cfg.law in _LJC_LAWS else None
        if gv is not None and bool(torch.any(gv != 0)):
            api.adjoint(pos_T, lam_v, ctx.prm, law=cfg.law, G=cfg.G, eps=cfg.eps,
                        alpha=0.5 * cfg.dt, grad_x=lam_x, grad_m=grad_m, grad_types=gt,
                        ntypes=cfg.ntypes, accumulate=True)
        nck = len(ctx.chunks)
        starts = [cfg.k * c for c in range(nck)]
        main = torch.cuda.current_stream(dev)
        side = None
        if any(ckpt is not None for _, ckpt in ctx.chunks):
            side = _side_stream(dev)
            side.wait_stream(main)  # checkpoints and prm were written on the main stream
        side_acc = []

        def positions(c):
            """Chunk c's positions and, where they are recomputed, the event after which
            they are there: enqueued on the side stream.
            The sweep reads x_0 .. x_{steps-1} of the chunk: steps - 1 leapfrog
            steps from the checkpoint (with its stored a(x_0) where the forward pass
            carried one in) give exactly those, with the forward's own kernels and
            bits, and no force evaluation whose result the sweep does not use."""
            if ctx.chunks[c][0] is not None:
                return ctx.chunks[c][0], None
            p0, v0, l0, a0 = ctx.chunks[c][1]
            steps = min(cfg.k, cfg.nsteps - starts[c])
            with torch.cuda.stream(side):
                pos, vel, lo = p0.clone(), v0.clone(), l0.clone()
                if not side_acc:
                    side_acc.append(torch.empty_like(pos))
                if a0 is not None:
                    side_acc[0].copy_(a0)
                trace = torch.empty((steps * n, 4), dtype=torch.float32, device=dev)
                api.step(pos, vel, side_acc[0], ctx.prm, dt=cfg.dt, nsteps=steps - 1,
                         law=cfg.law, G=cfg.G, eps=cfg.eps, acc_valid=a0 is not None,
                         trace=trace, state_lo=lo, stream=side)
            done = torch.cuda.Event()
            done.record(side)
            return trace, done

        pending = positions(nck - 1) if nck else None
        for c in range(nck - 1, -1, -1):
            steps = min(cfg.k, cfg.nsteps - starts[c])
            trace, done = pending
            if done is not None:
                main.wait_event(done)
                trace.record_stream(main)
            pending = positions(c - 1) if c > 0 else None
            api.adjoint_leapfrog(trace, lam_x, lam_v, ctx.prm, k=steps, dt=cfg.dt,
                                 first=starts[c] == 0, law=cfg.law, G=cfg.G, eps=cfg.eps,
                                 grad_m=grad_m, grad_types=gt, ntypes=cfg.ntypes, stream=main)
        g_sig = g_eps = None
        if cfg.law in _LJC_LAWS:
            g_sig = grad_t[:cfg.ntypes].to(torch.float32)
            g_eps = grad_t[cfg.ntypes:].to(torch.float32)
        return lam_x[:, :3].clone(), lam_v[:, :3].clone(), grad_m, g_sig, g_eps, None


def leapfrog(x0, v0, m, *, dt, nsteps, k=20, G=1.0, eps=0.0, law=LAW_GRAV, q=None,
             types=None, sig_t=None, eps_t=None, kq=None, keep_bytes=None):
    """Differentiable leapfrog: returns (x_T, v_T); gradients flow to x0, v0, m
    and (LJC) sig_t, eps_t. Gravity by default; pass law=LAW_LJC (or
    LAW_LJC_LINEAR, the linear dielectric) with per-atom charges q (float64),
    int32 types and per-type sig_t, eps_t for LJ + Coulomb; kq defaults to
    k_e / 80 (constant) or k_e / 4 (linear, dielectric 4 r).

    Positions between the forward and the backward pass: those of the newest ``k`` steps and
    as many more as fit in ``keep_bytes`` (0: no more; None: 32 MiB, or up to a 256th of the
    device's memory and a 64th of what is free); the older chunks of k steps are recomputed
    from checkpoints. The gradients are the same."""
    if law in _LJC_LAWS:
        if kq is None:
            kq = api.COULOMB_K / (80.0 if law == LAW_LJC else 4.0)
        ntypes = int(sig_t.shape[0])
        cfg = _Cfg(law, dt, nsteps, k, G, eps, q=q, types=types, kq=kq, ntypes=ntypes,
                   keep_bytes=keep_bytes)
    else:
        cfg = _Cfg(law, dt, nsteps, k, G, eps, keep_bytes=keep_bytes)
        sig_t = eps_t = torch.zeros(0, device=x0.device)
    return NBodyLeapfrog.apply(x0, v0, m, sig_t, eps_t, cfg)
