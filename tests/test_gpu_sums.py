"""Rounding of the sums of the kernels that default calls run: against 64 bits their rms
error is no larger than that of the tile that the stored table names for the size, on the
same inputs. The bound allows for 3%, the spread of an rms over some thousand particles."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from gpu_util import dev, floored_errors, grav_tensors, lib

pytestmark = pytest.mark.gpu

SPREAD = 1.03


def _rms(e):
    return float(np.sqrt(np.mean(e * e)))


def _compare(kinds, ref, floor=0.05):
    """kinds: outputs of the default call and of the tile."""
    own, tile = (_rms(floored_errors(k.cpu().numpy(), ref, floor)) for k in kinds)
    assert own <= SPREAD * tile, f"rms error {own:.3e}, tile {tile:.3e}"


@pytest.mark.parametrize("n", [4001, 8192, 12287, 32769])
def test_forces_and_potential(n):
    nb = lib()
    g = workloads.plummer(n, seed=n, eps=0.01)
    pos, _ = grav_tensors(g)
    eps = float(np.float32(g.eps))
    x, _, m = g.f32_as_f64()
    ref, phi = oracle.grav_accel(x, m, eps=eps, potential=True)
    tile, js = nb.get_config(nb.LAW_GRAV, n)
    out = [nb.forces(pos, eps=eps, pot=True, **kw) for kw in ({}, dict(tile=tile, jsplit=js))]
    _compare([o[:, :3] for o in out], ref)
    _compare([o[:, 3] for o in out], phi)
    assert torch.equal(out[0][:, :3], nb.forces(pos, eps=eps)[:, :3])


@pytest.mark.parametrize("n", [20001, 65536])
def test_subset(n):
    """Four lists of 2000 active particles."""
    nb = lib()
    g = workloads.plummer(n, seed=n, eps=0.01)
    pos, _ = grav_tensors(g)
    eps = float(np.float32(g.eps))
    x, _, m = g.f32_as_f64()
    idx = np.random.default_rng(n).permutation(n)[:8000].astype(np.int32)
    ref = oracle.grav_accel(x, m, eps=eps, idx=idx)
    tile, js = nb.get_config(nb.LAW_GRAV, 2000)
    out = [torch.cat([nb.forces_subset(pos, torch.from_numpy(k).to(dev()), eps=eps, **kw)
                      for k in np.split(idx, 4)]) for kw in ({}, dict(tile=tile, jsplit=js))]
    _compare([o[:, :3] for o in out], ref)


@pytest.mark.parametrize("n", [5000, 6500])
def test_gravity_vjp(n):
    nb = lib()
    errs = []
    for seed in range(4):
        g = workloads.plummer(n, seed=seed, eps=0.01)
        pos, _ = grav_tensors(g)
        eps = float(np.float32(g.eps))
        x, _, m = g.f32_as_f64()
        lam = np.random.default_rng(seed).standard_normal((n, 4)).astype(np.float32)
        tl = torch.from_numpy(lam).to(dev())
        rg, rm = oracle.grav_vjp(x, m, lam[:, :3].astype(np.float64), eps=eps)
        tile, js = nb.get_config(nb.TABLE_VJP_GRAV, n)
        row = []
        for kw in ({}, dict(tile=tile, jsplit=js)):
            gx, gm, _ = nb.adjoint(pos, tl, eps=eps, **kw)
            row += [_rms(floored_errors(gx[:, :3].cpu().numpy(), rg, 0.05)),
                    _rms(floored_errors(gm.cpu().numpy(), rm, 0.05))]
        errs.append(row)
    gx, gm, tx, tm = np.sqrt(np.mean(np.square(errs), 0))
    assert gx <= SPREAD * tx and gm <= SPREAD * tm, f"{gx:.3e} {tx:.3e}, {gm:.3e} {tm:.3e}"
