"""Local criteria at doses whose squared tolerance is below the smallest float
(Delta D of 3 % of 1e-24): where both doses agree gamma is 0, not 0 / 0."""
import numpy as np
import pytest

import synth
from tests.test_gpu_parity import assert_parity, gpu_gamma, oracle_gamma

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walk", [3, 0, 1])
@pytest.mark.parametrize("shape", [(3, 40), (9, 33), (2, 3, 34), (5, 6, 37)], ids=str)
def test_equal_tiny_doses_have_gamma_zero(shape, walk):
    rng = np.random.default_rng(sum(shape))
    ref = rng.uniform(0.5, 1.0, shape).astype(np.float32)
    ev = (ref * rng.uniform(0.98, 1.02, shape)).astype(np.float32)
    half = shape[-1] // 2
    ref[..., :half] = ev[..., :half] = 1e-24
    # one tiny voxel among ordinary ones, and one ordinary voxel among tiny ones
    ref[(0,) * (len(shape) - 1) + (half + 3,)] = ev[(0,) * (len(shape) - 1) + (half + 3,)] = 1e-24
    ref[(1,) * (len(shape) - 1) + (2,)] = ev[(1,) * (len(shape) - 1) + (2,)] = 0.75
    c = synth.Criteria(0.03, 2.0, local=True, cutoff_frac=0.0)
    sp = (1.5, 1.0, 1.0)[3 - len(shape):]
    got, counts, _ = gpu_gamma(ref, ev, sp, c, {"walk": walk})
    assert (got[..., :half] == 0).all()
    assert_parity(got, oracle_gamma(ref, ev, sp, c), counts)
