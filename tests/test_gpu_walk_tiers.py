"""The warp-evaluated walk (plane seeds, dose gap, plane bound, faces) at the
sizes where its parts can go wrong: grids of two or three voxels per axis
(every cell at the grid's edge, seeds clamped to it), rows that do not fill a
warp, tables cut short (voxels left to the finishing pass), one to 32 lanes
per voxel, and queues shorter and longer than the resident warps.

Every cell is evaluated with the arithmetic of the lane walk (option walk =
0) and a cell is only passed over when it cannot hold the nearest point, so
the two maps are equal bit for bit; the oracle bounds both.
"""
import numpy as np
import pytest

import synth
from tests.test_gpu_parity import assert_parity, gpu_gamma, oracle_gamma

pytestmark = pytest.mark.gpu


def _pair(shape, seed, smooth):
    rng = np.random.default_rng(seed)
    ref = rng.uniform(0.2, 1.0, shape)
    ev = rng.uniform(0.2, 1.0, shape)
    if smooth:                                   # planes with a little curvature: seeds near the foot
        c = np.meshgrid(*[np.linspace(0, 1, n) for n in shape], indexing="ij")
        ref = 0.5 + 0.3 * sum(c) / len(c) + 0.02 * c[-1] ** 2
        ev = ref + 0.05 + 0.03 * np.sin(3 * c[0])
    return ref.astype(np.float32), ev.astype(np.float32)


@pytest.mark.parametrize("opt", [{}, {"group_bucket": 32}, {"group_bucket": 0, "group8_bucket": 3, "group32_bucket": 6},
                                 {"table_cap": 24}, {"sort_tail": 0}], ids=["default", "lane", "tiers", "cut", "unsorted"])
@pytest.mark.parametrize("crit", [(0.03, 3.0, False), (0.01, 1.0, True)], ids=["3-3", "1-1-local"])
@pytest.mark.parametrize("smooth", [False, True], ids=["noise", "smooth"])
@pytest.mark.parametrize("shape", [(2, 2, 2), (2, 3, 37), (5, 33, 34), (2, 2), (3, 70), (65, 47)], ids=str)
def test_tiered_walk_is_bitwise_the_lane_walk(shape, smooth, crit, opt):
    ref, ev = _pair(shape, sum(shape), smooth)
    sp = (1.0, 2.0, 1.5)[3 - len(shape):]
    c = synth.Criteria(crit[0], crit[1], local=crit[2])
    lane = {k: v for k, v in opt.items() if k in ("table_cap", "sort_tail")}
    a, ca, sa = gpu_gamma(ref, ev, sp, c, dict(lane, walk=0))
    b, cb, sb = gpu_gamma(ref, ev, sp, c, dict(opt, walk=3))
    np.testing.assert_array_equal(a, b)
    assert ca == cb and sa["tail_voxels"] == sb["tail_voxels"]
    assert_parity(b, oracle_gamma(ref, ev, sp, c), cb)


def test_long_queue_takes_whole_batches_of_rounds():
    # more queued voxels than the resident warps hold, so that batches run
    # several rounds; thin slab: edge cells on every voxel's walk
    p = synth.make_pair_3d(shape=(3, 320, 300), spacing=(1.25, 1.25, 1.25), seed=11, shift_mm=(0.0, 1.0, 3.0),
                           scale=1.05, criteria=synth.Criteria(0.02, 3.0, cutoff_frac=0.0))
    a, ca, _ = gpu_gamma(p.ref, p.eval, p.spacing, p.criteria, {"walk": 0})
    b, cb, sb = gpu_gamma(p.ref, p.eval, p.spacing, p.criteria, {"walk": 3})
    assert sb["tail_voxels"] > 100000
    np.testing.assert_array_equal(a, b)
    assert ca == cb


@pytest.mark.parametrize("shape", [(17, 33, 31), (16, 20, 32), (34, 18, 63), (2, 40, 65), (90, 62), (47, 130)], ids=str)
def test_costly_queue_reads_dose_ranges(shape):
    # a dose offset of many gamma: hundreds of tested cells per voxel of the
    # grid, far past the line where the cells' dose ranges come from an array;
    # rows and columns around the 31 cells and 16 planes of its pass
    rng = np.random.default_rng(sum(shape))
    ref = rng.uniform(0.5, 0.6, shape).astype(np.float32)
    ev = rng.uniform(0.7, 0.9, shape).astype(np.float32)
    sp = (1.0, 1.5, 1.25)[3 - len(shape):]
    c = synth.Criteria(0.03, 1.5)
    a, ca, sa = gpu_gamma(ref, ev, sp, c, {"walk": 0, "stats": 1})
    b, cb, sb = gpu_gamma(ref, ev, sp, c, {"walk": 3, "stats": 1})
    assert sb["cells_keyed"] > 12 * ref.size
    np.testing.assert_array_equal(a, b)
    assert ca == cb
    assert_parity(b, oracle_gamma(ref, ev, sp, c), cb)
