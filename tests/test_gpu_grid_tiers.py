"""The two-grid search (plane seeds, tiered walk) over the forms it takes:
evaluation grids of two nodes on an axis (every cell at an edge), reference
points far outside the evaluation grid, single-voxel reference axes, coarser
and finer evaluation grids, and every lane count.

The number of lanes only changes the order in which cells are looked at, and
a cell is passed over only when it cannot hold the nearest point, so the maps
agree bit for bit; the oracle bounds them (1e-4)."""
import numpy as np
import pytest

import synth
from tests.test_gpu_grids import check, gpu_grids, oracle_grids

pytestmark = pytest.mark.gpu

CASES = {
    "two_nodes": ((3, 4, 5), (1.0, 1.1, 0.9), (0.2, 0.1, 0.3), (2, 2, 2), (2.5, 2.0, 3.0), (0.0, 0.0, 0.0)),
    "outside": ((4, 5, 6), (2.0, 2.0, 2.0), (-9.0, 11.0, -7.0), (6, 7, 5), (1.5, 1.25, 2.0), (0.0, 0.0, 0.0)),
    "one_row": ((1, 1, 40), (1.0, 1.0, 0.7), (3.1, 2.9, -1.0), (5, 6, 21), (1.5, 1.25, 1.3), (0.0, 0.0, 0.0)),
    "coarser": ((12, 13, 14), (1.0, 1.0, 1.0), (0.5, 0.25, 0.75), (5, 6, 7), (3.0, 2.5, 2.0), (0.0, 0.0, 0.0)),
    "finer": ((7, 8, 9), (2.5, 2.5, 2.5), (0.6, 0.3, 0.9), (20, 21, 33), (1.0, 1.0, 0.75), (-0.5, 0.0, 0.0)),
    "plane": ((17, 35), (1.3, 0.8), (-2.0, 1.0), (16, 41), (1.0, 1.0), (0.0, 0.0)),
}


def _doses(name, seed):
    rshape, rsp, ro, eshape, esp, eo = CASES[name]
    rng = np.random.default_rng(seed)

    def field(shape, sp, o, scale):
        x = np.meshgrid(*[a + h * np.arange(n) for n, h, a in zip(shape, sp, o)], indexing="ij")
        f = 0.6 + 0.2 * np.sin(0.25 * x[-1]) + 0.15 * np.cos(0.3 * x[0] + 0.2 * x[-2])
        return (scale * f + rng.normal(0, 0.01, shape)).astype(np.float32)

    return field(rshape, rsp, ro, 1.0), field(eshape, esp, eo, 1.04)


@pytest.mark.parametrize("crit", [(0.02, 2.0, False), (0.01, 1.0, True)], ids=["2-2", "1-1-local"])
@pytest.mark.parametrize("name", list(CASES))
def test_lane_counts_agree_and_match_the_oracle(name, crit):
    rshape, rsp, ro, eshape, esp, eo = CASES[name]
    ref, ev = _doses(name, 3)
    c = synth.Criteria(crit[0], crit[1], local=crit[2])
    want = oracle_grids(ref, rsp, ro, ev, esp, eo, c)
    first = None
    for opt in ({}, {"lanes_per_voxel": 2}, {"lanes_per_voxel": 32}, {"walk": 3, "lanes_per_voxel": 16},
                {"table_cap": 40, "lanes_per_voxel": 4}):
        got, counts, _ = gpu_grids(ref, rsp, ro, ev, esp, eo, c, opt)
        check(got, want, counts)
        first = got if first is None else first
        np.testing.assert_array_equal(got, first)
