"""Batches of planes and volumes, whose two groups run side by side: the run
ends on the caller's stream only when both have.  A consumer queued right
after it on that stream, with no host synchronisation in between, sees the
finished maps of both groups, and the next run may overwrite them."""
import numpy as np
import pytest

from tests.test_gpu_batch import _batch_run, _pairs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("own_stream", [False, True])
@pytest.mark.parametrize("graph", [0, 1])
def test_both_groups_end_on_the_callers_stream(graph, own_stream):
    import paper_1012_1900_gb300 as g
    ps = _pairs()
    want = _batch_run(ps, {"timing": 1})[0][0][0]        # one stream throughout
    s = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
    with torch.cuda.stream(s):
        data = [(torch.from_numpy(p.ref).cuda(), torch.from_numpy(p.eval).cuda()) for p in ps]
        outs = [torch.empty_like(r) for r, _ in data]
        descs = []
        for p, (r, e), o in zip(ps, data, outs):
            nd, c = p.ref.ndim, p.criteria
            descs.append((r, e, o, nd, p.ref.shape if nd == 3 else (1,) + p.ref.shape,
                          p.spacing if nd == 3 else (1.0,) + p.spacing,
                          g.criteria(c.dd_frac, c.dta_mm, c.local, c.cutoff_frac, c.dose_norm)))
        h = g.gamma_batch_create(descs)
        try:
            g.gamma_set_option(h, "graph", graph)
            got = []
            for _ in range(3):
                for o in outs:
                    o.fill_(-7.0)
                g.gamma_batch_run(h, s)
                got.append([o.clone() for o in outs])
            s.synchronize()
        finally:
            g.gamma_destroy(h)
    for maps in got:
        for a, b in zip(maps, want):
            np.testing.assert_array_equal(a.cpu().numpy().astype(np.float64), b)
