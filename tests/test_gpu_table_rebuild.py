"""A table that finds no room on the device (option table_cap) is refused, and
the handle goes on with the one that it has."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_refused_table_leaves_the_old_one():
    import paper_1012_1900_gb300 as g
    p = synth.make_pair_3d(shape=(96, 128, 128), spacing=(2.5, 2.5, 2.5), seed=5, shift_mm=(0.5, 1.0, 1.0), scale=1.02)
    r, e = torch.from_numpy(p.ref).cuda(), torch.from_numpy(p.eval).cuda()
    out = torch.empty_like(r)
    h = g.gamma_create(r, e, 3, p.ref.shape, p.spacing, g.criteria(0.03, 3.0))
    try:
        g.gamma_run(h, out)
        counts, entries = g.gamma_pass_rate(h), g.gamma_get_stats(h)["table_entries"]
        want = out.cpu().numpy()
        torch.cuda.empty_cache()
        # room for 64 MiB; the table of 4 M cells takes 96 MiB
        rest = torch.cuda.mem_get_info()[0] - (64 << 20)
        fill = torch.empty(rest, dtype=torch.uint8, device="cuda")
        try:
            with pytest.raises(g.GammaError) as err:
                g.gamma_set_option(h, "table_cap", 1 << 22)
            assert err.value.code == -4                      # GAMMA_ERR_OOM
        finally:
            del fill
            torch.cuda.empty_cache()
        out.fill_(-7.0)
        g.gamma_run(h, out)
        assert g.gamma_pass_rate(h) == counts and g.gamma_get_stats(h)["table_entries"] == entries
        np.testing.assert_array_equal(out.cpu().numpy(), want)
        g.gamma_set_option(h, "table_cap", 1 << 22)          # with room it is taken
        g.gamma_run(h, out)
        assert g.gamma_pass_rate(h) == counts and g.gamma_get_stats(h)["table_entries"] > entries
        np.testing.assert_array_equal(out.cpu().numpy(), want)
    finally:
        g.gamma_destroy(h)
