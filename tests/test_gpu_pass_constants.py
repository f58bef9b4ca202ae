"""The 3-pass form's sweep constants come from a table that follows dt: captured sequences
replayed with another dt, both pass kernels (blocks on one side of v = 0 and across it), and
the two forms, whose values must be the same bits."""
import numpy as np
import pytest

from paper_2504_21450_gb300 import inputs, vlasov

pytestmark = pytest.mark.gpu


def run(n, nv, vmin, dts, form, graph, storage=vlasov.VL_STORE_F32):
    init = inputs.random_blocks(n, nv, 1.0, seed=106)
    g = vlasov.Grid(n, nv, vmin, (0.7, 0.9, 1.1), storage=storage)
    g.set_blocks(init.off, init.ids, init.vals)
    for dt in dts:
        g.translate(dt, "xyz", 2, form=form, graph=graph)
    out = g.get_blocks()
    g.close()
    return out


@pytest.mark.parametrize("vmin", [(-2.8, -3.6, -4.4), (-2.1, -3.6, -4.4)])
def test_captured_passes_follow_dt(vmin):
    dts = (0.05, 0.11, 0.05)
    want = run((9, 8, 7), (8, 8, 8), vmin, dts, vlasov.VL_FORM_3PASS, False)
    got = run((9, 8, 7), (8, 8, 8), vmin, dts, vlasov.VL_FORM_3PASS, True)
    for a, b in zip(want, got):
        assert np.array_equal(a, b)


def test_forms_agree():
    args = ((20, 17, 9), (8, 8, 8), (-2.8, -3.6, -4.4), (0.037, 0.113))
    want = run(*args, vlasov.VL_FORM_FUSED, False)
    got = run(*args, vlasov.VL_FORM_3PASS, False)
    for a, b in zip(want, got):
        assert np.array_equal(a, b)
