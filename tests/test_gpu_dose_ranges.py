"""The cells' dose ranges on costly queues: the ordering pass that writes them
tells the walk so, and the walk reads them only then.  Without that pass
(option sort_tail = 0), and on a handle whose inputs change between runs, the
map has to be the lane walk's (option walk = 0) bit for bit.
"""
import numpy as np
import pytest

from tests.test_gpu_parity import gpu_gamma

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CRIT = synth.Criteria(0.03, 1.5)


def _pair(shape, seed, offset):
    # an offset of many gamma: hundreds of tested cells per voxel of the grid
    rng = np.random.default_rng(seed)
    ref = rng.uniform(0.5, 0.6, shape).astype(np.float32)
    return ref, (rng.uniform(0.5, 0.7, shape) + offset).astype(np.float32)


def _spacing(shape):
    return (1.0, 1.5, 1.25)[3 - len(shape):]


@pytest.mark.parametrize("shape", [(17, 33, 31), (16, 20, 32), (90, 62)], ids=str)
def test_unordered_queue_reads_no_ranges(shape):
    ref, ev = _pair(shape, sum(shape), 0.2)
    want, cw, _ = gpu_gamma(ref, ev, _spacing(shape), CRIT, {"walk": 0})
    got, cg, _ = gpu_gamma(ref, ev, _spacing(shape), CRIT, {"sort_tail": 0})
    np.testing.assert_array_equal(want, got)
    assert cw == cg


def test_ranges_are_those_of_the_run():
    # costly, costly with other doses, cheap, unordered, costly: one handle
    import paper_1012_1900_gb300 as g
    shape = (17, 33, 31)
    steps = [(1, 0.2, 1), (2, -0.2, 1), (3, 0.0, 1), (4, 0.25, 0), (5, 0.15, 1)]
    h, tensors = None, []
    try:
        for seed, offset, order in steps:
            ref, ev = _pair(shape, seed, offset)
            want, cw, _ = gpu_gamma(ref, ev, _spacing(shape), CRIT, {"walk": 0})
            r, e = torch.from_numpy(ref).cuda(), torch.from_numpy(ev).cuda()
            out = torch.full_like(r, -7.0)
            tensors += [r, e, out]
            if h is None:
                h = g.gamma_create(r, e, 3, shape, _spacing(shape), g.criteria(CRIT.dd_frac, CRIT.dta_mm))
            g.gamma_set_inputs(h, r, e)
            g.gamma_set_option(h, "sort_tail", order)
            for _ in range(3):                               # direct, direct, replayed
                g.gamma_run(h, out)
                assert g.gamma_pass_rate(h) == cw
                np.testing.assert_array_equal(want, out.cpu().numpy().astype(np.float64))
    finally:
        g.gamma_destroy(h)
