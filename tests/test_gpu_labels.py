"""Labels (one warp per voxel, pruned) where their rounds and bounds can go
wrong: planes, slabs two voxels thick (every cell at the grid's edge), more
listed voxels than warps, and a map that does not hold the distances of its
own search (the pruning then has nothing to go by).

A label's point must lie on the evaluation surface at the distance the gamma
map holds: the two differ by FP32 rounding of coordinates up to a few units
and doses of order one over Delta D, 2e-4 at most for the criteria here.
"""
import math

import numpy as np
import pytest

import synth
from tests import _brute as brute

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _labels(p, crit, scale=1.0, reps=1):
    import paper_1012_1900_gb300 as g
    nd = p.ref.ndim
    shape = p.ref.shape if nd == 3 else (1,) + p.ref.shape
    sp = tuple(p.spacing) if nd == 3 else (1.0,) + tuple(p.spacing)
    r, e = torch.from_numpy(p.ref).cuda(), torch.from_numpy(p.eval).cuda()
    out = torch.empty_like(r)
    h = g.gamma_create(r, e, nd, shape, sp, g.criteria(crit.dd_frac, crit.dta_mm, crit.local, crit.cutoff_frac))
    try:
        g.gamma_run(h, out)
        g.gamma_pass_rate(h)
        gm = out.cpu().numpy().ravel().astype(np.float64)
        vox = np.tile(np.arange(p.ref.size, dtype=np.int32), reps)
        T = torch.empty((vox.size, 4), device="cuda")
        g.gamma_labels(h, out * scale, torch.from_numpy(vox).cuda(), T)
        T = T.cpu().numpy().astype(np.float64)
    finally:
        g.gamma_destroy(h)
    return gm, T


def _distances(p, crit, T, vox):
    hn = np.array(p.spacing[::-1]) / crit.dta_mm
    out = []
    for v in vox:
        idx = np.array(np.unravel_index(v, p.ref.shape), dtype=np.float64)
        pos = idx + (T[v, :p.ref.ndim] / hn)[::-1]
        de = brute.freudenthal_interpolate(p.eval, pos[::-1][None, :])[0]
        dr = float(p.ref.ravel()[v])
        dD = float(np.float32(crit.dd_frac)) * (dr if crit.local else float(p.ref.max()))
        out.append(math.sqrt(float((T[v, :3] ** 2).sum()) + ((de - dr) / dD) ** 2))
    return np.array(out)


@pytest.mark.parametrize("local", [False, True], ids=["global", "local"])
@pytest.mark.parametrize("shape", [(23, 37), (2, 19, 33), (11, 12, 13)], ids=str)
def test_labels_lie_on_the_surface_at_the_map_s_distance(shape, local):
    crit = synth.Criteria(0.02, 2.0, local=local, cutoff_frac=0.1)
    make = synth.make_pair_2d if len(shape) == 2 else synth.make_pair_3d
    shift = (0.0, 1.5, 2.0)[3 - len(shape):]
    p = make(shape=shape, spacing=(2.0, 1.5, 1.25)[3 - len(shape):], seed=5, shift_mm=shift, scale=1.04, criteria=crit)
    gm, T = _labels(p, crit)
    ok = np.isfinite(gm)
    assert np.array_equal(np.isfinite(T[:, 3]), ok) and ok.any()
    vox = np.nonzero(ok)[0]
    np.testing.assert_allclose(_distances(p, crit, T, vox), gm[vox], rtol=0, atol=2e-4)
    np.testing.assert_allclose(T[vox, 3], np.log(gm[vox] + 1e-3), rtol=0, atol=1e-4)


def test_labels_do_not_depend_on_the_list_or_on_a_scaled_map():
    crit = synth.Criteria(0.02, 2.0)
    p = synth.make_pair_3d(shape=(9, 20, 24), spacing=(2.0, 2.0, 2.0), seed=6, shift_mm=(0.0, 1.0, 2.5), scale=1.04,
                           criteria=crit)
    gm, T = _labels(p, crit)
    gm2, T2 = _labels(p, crit, reps=5)
    np.testing.assert_array_equal(T2, np.tile(T, (5, 1)))
    # a map scaled by 1.5 only widens the search: the same points
    _, T3 = _labels(p, crit, scale=1.5)
    ok = np.isfinite(gm)
    np.testing.assert_array_equal(T3[ok, :3], T[ok, :3])
    # a map scaled by 0.97 says less than any distance: still the nearest of the cells it reaches
    _, T4 = _labels(p, crit, scale=0.97)
    d = _distances(p, crit, T4, np.nonzero(ok)[0])
    assert np.all(d >= gm[ok] - 2e-4)
