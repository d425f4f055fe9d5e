"""The training pass (rows' kernel and weight gradients) where its tiles end:
one row, fewer rows than a column group of the transposed operands, one tile
less and more than full, a batch after a larger one (the workspace keeps its
larger rows), element by element against the FP64 reference with the same bf16
rounding points (bounds of tests/_nnbound.py)."""
import numpy as np
import pytest

from oracle import mlp
from tests import _nnbound as nb
from tests.test_gpu_learned import _bf16_rows

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sizes", [(1,), (7,), (127,), (128,), (129,), (640, 63)], ids=str)
def test_gradients_of_ragged_batches(sizes):
    import paper_1012_1900_gb300 as g
    rng = np.random.default_rng(sum(sizes))
    m = g.gamma_model_create(17)
    try:
        p = g.gamma_model_get_params(m).astype(np.float64)
        for M in sizes:
            Xb, Xq = _bf16_rows(rng, M)
            T = rng.normal(0, 1, (M, 4)).astype(np.float32)
            if M > 5:
                T[3, 3] = np.nan
            loss = g.gamma_model_backward(m, Xb, torch.from_numpy(T).cuda())
            want_loss, want_g, e_loss, e_g = nb.backward_bounds(p, Xq, T)
            assert abs(loss - want_loss) <= e_loss + 1e-7
            got = g.gamma_model_get_params(m, which=1).astype(np.float64)
            assert np.all(got[~mlp.trainable_mask()] == 0)
            assert np.all(np.abs(got - want_g) <= e_g + 1e-12)
    finally:
        g.gamma_model_destroy(m)
