"""Device memory of a handle and what it does with less of it: the bytes per
voxel that gamma.h names, and maps that do not depend on the optional lists
(the option that runs without them takes the same branches as a failed
allocation)."""
import numpy as np
import pytest

import synth
from tests.test_gpu_parity import assert_parity, gpu_gamma, oracle_gamma

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SLACK = 24 << 20        # tables (3 MiB per pair), allocation granularity, a stream's own memory


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _doses(n, shape):
    return [tuple(torch.rand(shape, device="cuda") for _ in range(3)) for _ in range(n)]


def test_scratch_per_voxel():
    import paper_1012_1900_gb300 as g
    shape = (128, 256, 256)
    nvox = 128 * 256 * 256
    crit = g.criteria(0.03, 3.0)
    pairs = _doses(2, shape)
    sp = (1.0, 1.0, 1.0)
    g.gamma_destroy(g.gamma_create(*pairs[0][:2], 3, shape, sp, crit))
    before = _free()
    h = g.gamma_create(*pairs[0][:2], 3, shape, sp, crit)
    single = before - _free()
    g.gamma_destroy(h)
    assert single <= 29 * nvox + SLACK
    g.gamma_destroy(g.gamma_batch_create([(r, e, o, 3, shape, sp, crit) for r, e, o in pairs]))
    before = _free()
    h = g.gamma_batch_create([(r, e, o, 3, shape, sp, crit) for r, e, o in pairs])
    batch = before - _free()
    g.gamma_destroy(h)
    assert batch <= 2 * (25 * nvox + SLACK)


@pytest.mark.parametrize("extra", [{}, {"sort_tail": 0}, {"graph": 0}, {"table_cap": 64}], ids=str)
@pytest.mark.parametrize("drop", [1, 2])
@pytest.mark.parametrize("shape", [(17, 33, 31), (90, 62)], ids=str)
def test_maps_do_not_depend_on_optional_lists(shape, drop, extra):
    # a costly queue, so that the full handle reads dose ranges
    rng = np.random.default_rng(sum(shape))
    ref = rng.uniform(0.5, 0.6, shape).astype(np.float32)
    ev = rng.uniform(0.7, 0.9, shape).astype(np.float32)
    sp = (1.0, 1.5, 1.25)[3 - len(shape):]
    c = synth.Criteria(0.03, 1.5)
    full, cf, _ = gpu_gamma(ref, ev, sp, c, extra, runs=3)
    less, cl, _ = gpu_gamma(ref, ev, sp, c, dict(extra, drop_lists=drop), runs=3)
    for a, b in zip(full, less):
        np.testing.assert_array_equal(a, b)
    assert cf == cl
    if not extra:
        assert_parity(less[0], oracle_gamma(ref, ev, sp, c), cl)
