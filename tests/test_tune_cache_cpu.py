"""The tuning cache: entries that were installed before the kernels of default calls come back
as such, the others as stored ones."""
import json

import torch

from paper_0706_3060_gb300 import _lib, api, tune


def test_installed_and_stored_entries(tmp_path, monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_available", lambda: True)
    monkeypatch.setattr(tune, "_gpu_key", lambda torch: "test")
    lib = api._lib()
    buckets = (40, 41, 42)  # of sizes that nobody has
    path = tmp_path / "cache.json"
    ent = {"n": 0, "tile": 1, "jsplit": 0, "ms": 1.0}
    path.write_text(json.dumps({"test": {"0": {"40": ent, "41": dict(ent, installed=True)}}}))
    try:
        assert tune.load_cache(str(path)) == 2
        assert [lib.nbody_tuned_kind(0, b) for b in buckets] == [1, 2, 0]
        # what is saved is what is loaded again
        table = {str(b): tune._entry(0, b, 1 << b, 1, 0, 1.0) for b in (40, 41)}
        tune.save_cache(0, table, str(path))
        for b in buckets:
            tune._install(0, b, -1, 0, False)
        assert tune.load_cache(str(path)) == 2
        assert [lib.nbody_tuned_kind(0, b) for b in buckets] == [1, 2, 0]
    finally:
        for b in buckets:
            tune._install(0, b, -1, 0, False)
    assert lib.nbody_tuned_kind(0, 64) == -1 and lib.nbody_tuned_kind(99, 1) == -1
    assert "nbody_tuned_kind" in _lib.EXPORTS
