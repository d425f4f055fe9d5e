"""The blocks that the passes over a batch's queues take per pair: pairs of one
block (up to 256 voxels), of one voxel more, and of more blocks than a pair
gets at most (four per SM), so that its blocks take several turns.  Every
voxel is queued; the maps are those of one run per pair."""
import numpy as np
import pytest

import synth
from tests.test_gpu_batch import _batch_run
from tests.test_gpu_parity import gpu_gamma

pytestmark = pytest.mark.gpu


def _pair(shape, seed):
    rng = np.random.default_rng(seed)
    ref = rng.uniform(0.5, 0.6, shape).astype(np.float32)
    ev = (rng.uniform(0.5, 0.6, shape) + 0.06).astype(np.float32)
    return synth.Pair("noise", ref, ev, (1.5,) * len(shape), synth.Criteria(0.03, 2.0))


@pytest.mark.parametrize("shapes", [[(2, 2, 2), (4, 8, 8), (4, 8, 9), (64, 64, 80), (5, 3, 17)],
                                    [(16, 16), (2, 129), (500, 640), (2, 2)],
                                    [(13, 19), (3, 4, 5), (31, 70), (8, 8, 8)]], ids=str)
def test_batch_blocks_cover_every_queue(shapes):
    ps = [_pair(s, 31 + k) for k, s in enumerate(shapes)]
    (first, second), _ = _batch_run(ps, runs=2)
    for k, p in enumerate(ps):
        want, counts, stats = gpu_gamma(p.ref, p.eval, p.spacing, p.criteria)
        assert stats["tail_voxels"] > 0.5 * p.ref.size
        for maps, cnt in (first, second):
            np.testing.assert_allclose(maps[k], want, rtol=0, atol=1e-6, equal_nan=True)
            assert cnt[k] == counts
