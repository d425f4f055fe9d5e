"""Counters of a two-grid run: the search has no key-0 phase, so that no voxel
is one that searched past it, however the walk queues its voxels."""
import numpy as np
import pytest

import synth
from tests.test_gpu_grids import gpu_grids

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opt", [{}, {"walk": 3, "lanes_per_voxel": 32}, {"table_cap": 40}], ids=str)
def test_two_grid_counters(opt):
    rng = np.random.default_rng(8)
    ref = rng.uniform(0.5, 0.6, (5, 17, 19)).astype(np.float32)
    ev = rng.uniform(0.5, 0.7, (6, 15, 21)).astype(np.float32)
    got, counts, st = gpu_grids(ref, (2.0, 2.0, 2.0), (0.3, 0.2, 0.7), ev, (2.5, 2.25, 2.0), (0.0, 0.0, 0.0),
                                synth.Criteria(0.02, 2.0), opt)
    assert st["tail_voxels"] == 0
    assert st["n_voxels"] == ref.size and st["n_eval"] == counts[1] == np.isfinite(got).sum()
    assert st["n_pass"] == counts[2] == (got <= 1).sum()
