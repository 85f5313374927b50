"""How many steps' positions the differentiable leapfrog keeps between its passes."""
import types

import pytest
import torch

from paper_0706_3060_gb300 import autograd

GIB = 1 << 30


@pytest.fixture
def memory(monkeypatch):
    m = types.SimpleNamespace(free=256 * GIB, total=280 * GIB, asked=0)

    def info(dev):
        m.asked += 1
        return m.free, m.total
    monkeypatch.setattr(torch.cuda, "mem_get_info", info)
    monkeypatch.setattr(torch.cuda, "memory_reserved", lambda dev: 0)
    monkeypatch.setattr(torch.cuda, "memory_allocated", lambda dev: 0)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    return m


def _rows(n, nsteps, k, **kw):
    """Float4 rows per particle that the forward pass leaves."""
    kept = autograd._kept_steps(n, nsteps, k, "cuda", **kw)
    rows, done = 0, 0
    while done < nsteps:
        steps = min(k, nsteps - done)
        rows += steps + 1 if nsteps - done <= kept else 5
        done += steps
    return rows


@pytest.mark.parametrize("nsteps,k", [(1, 1), (7, 2), (40, 10), (200, 5), (200, 20), (1000, 3)])
def test_no_bytes_is_what_checkpoints_take(memory, nsteps, k):
    chunks = -(-nsteps // k)
    checkpoints = 5 * chunks + k + 1  # and the newest chunk's positions
    assert _rows(1 << 20, nsteps, k, keep_bytes=0) <= checkpoints
    assert not memory.asked


def test_budget_and_free_memory(memory):
    n, nsteps, k = 1 << 20, 1000, 20
    row = 16 * n
    instead = 5 * -(-nsteps // k) + k + 1
    for keep in (0, GIB, 8 * GIB):
        assert _rows(n, nsteps, k, keep_bytes=keep) * row <= keep + instead * row
    assert _rows(n, nsteps, k) * row <= memory.total // 256 + instead * row
    memory.free = 16 * GIB
    assert _rows(n, nsteps, k) * row <= memory.free // 64 + instead * row
    memory.free = 0
    assert _rows(n, nsteps, k) <= instead
    # small runs keep everything and do not ask
    memory.asked = 0
    assert autograd._kept_steps(16384, 40, 10, "cuda") >= 40 and not memory.asked
