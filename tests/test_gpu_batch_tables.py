"""Batches whose pairs' cell tables differ in length: a warp of the batched walk
holds voxels of neighbouring pairs, and each lane has to stay in its own pair's
table while the others' walks go on (a 5x3x3 volume has 225 cells; a walk to
gamma 8 on a 24-cube of the same spacing tests 2,728).

A cell is only passed over when it cannot hold the nearest point, so the maps
are those of the lane walk (option walk = 0) bit for bit.
"""
import numpy as np
import pytest

import synth
from tests.test_gpu_batch import _batch_run

pytestmark = pytest.mark.gpu


def _pair(shape, seed, offset):
    rng = np.random.default_rng(seed)
    ref = rng.uniform(0.5, 0.6, shape).astype(np.float32)
    ev = (rng.uniform(0.5, 0.6, shape) + offset).astype(np.float32)
    return synth.Pair("offset", ref, ev, (1.0,) * len(shape), synth.Criteria(0.03, 1.0))


# voxel counts that are no multiple of a batch of rounds, so that the last
# voxels of one pair share a warp with the first of the next
@pytest.mark.parametrize("shapes", [[(5, 3, 3), (24, 24, 24)], [(24, 24, 24), (3, 2, 3), (19, 21, 23), (2, 2, 2)],
                                    [(5, 7), (60, 60)], [(61, 47), (2, 3), (33, 70), (3, 3), (5, 3, 3), (20, 20, 21)]],
                         ids=str)
@pytest.mark.parametrize("opt", [{}, {"group_bucket": 32}, {"group32_bucket": 0}, {"tail_blocks_per_sm": 3}], ids=str)
def test_lanes_stay_in_their_own_pairs_table(shapes, opt):
    ps = [_pair(s, 7 + k, 0.15 + 0.02 * k) for k, s in enumerate(shapes)]
    want, _ = _batch_run(ps, {"walk": 0})
    got, _ = _batch_run(ps, opt, runs=2)
    for maps, counts in got:
        for a, b in zip(want[0][0], maps):
            np.testing.assert_array_equal(a, b)
        assert counts == want[0][1]
