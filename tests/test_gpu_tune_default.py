"""Tuning leaves default calls with the direct and streamed kernels where these are faster."""
import math

import pytest
import torch

import workloads
from gpu_util import grav_tensors, lib

pytestmark = pytest.mark.gpu


@pytest.fixture
def entry(request):
    """(table, n) without an installed entry, and as it was afterwards."""
    table, n = request.param
    nb = lib()
    c = nb.api._lib()
    bucket = int(math.floor(math.log2(n)))
    kind, (tile, js) = c.nbody_tuned_kind(table, bucket), nb.get_config(table, n)
    c.nbody_set_stored(table, bucket, tile if kind else -1, js)
    yield table, n, bucket
    (c.nbody_set_tuned if kind == 2 else c.nbody_set_stored)(table, bucket, tile if kind else -1,
                                                             js)


# direct and streamed forces, streamed jerk; the fixed-point table, whose calls run the tile
@pytest.mark.parametrize("entry", [(0, 1500), (0, 9000), (7, 9000), (4, 9000)], indirect=True)
@pytest.mark.parametrize("native", [True, False])
def test_single(entry, native):
    nb = lib()
    from paper_0706_3060_gb300 import tune
    table, n, bucket = entry
    if table == 4 and not native:
        pytest.skip("tuned by the library only")
    pos, vel = grav_tensors(workloads.plummer(n, seed=n, eps=0.01))

    def call():
        if table == 7:
            return nb.forces_jerk(pos, vel, eps=0.01)[1]
        return nb.forces(pos, eps=0.01, fixed=table == 4)
    before = call()
    got = tune.tune(table, [n], reps=3, verbose=False, native=native,
                    tiles=None if native else [0, 1, 2])[str(bucket)]
    assert nb.api._lib().nbody_tuned_kind(table, bucket) == 1 and "installed" not in got
    assert nb.get_config(table, n) == (got["tile"], got["jsplit"])
    if table != 4:
        assert torch.equal(before, call())


@pytest.mark.parametrize("entry", [(3, 1)], indirect=True)
def test_batched(entry):
    nb = lib()
    from paper_0706_3060_gb300 import tune
    got = tune.tune_batched(reps=3, verbose=False)["0"]
    assert 0 <= got["tile"] < nb.tile_count(3) and "installed" not in got
    assert nb.api._lib().nbody_tuned_kind(3, 0) == 1
