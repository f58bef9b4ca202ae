"""3-pass steps on sparse states whose item tables ask for exactly 48 KiB of shared memory, the
most that a kernel gets unless its limit is raised, beside the few static bytes of list mode:
extents 5, 10, 11, 22 and 23 on the first pass (512 cells of pencils per item, two rank tables),
742 and 743 on a pass in place (one table).  Each case in a process of its own, since a
limit that one launch raises holds for later ones.  The values are the fused form's, bit for
bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2504_21450_gb300 import inputs, vlasov

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(n, nv, order):
    vlasov.load(build_if_missing=True)
    init = inputs.random_blocks(n, nv, 0.01, seed=110)
    out = []
    for form in (vlasov.VL_FORM_3PASS, vlasov.VL_FORM_FUSED):
        g = vlasov.Grid(n, nv, tuple(-0.5 * a for a in nv), (1.0,) * 3, threshold=0.05)
        g.set_blocks(init.off, init.ids, init.vals)
        g.translate(0.4 / max(nv), order, 1, form, check=True)
        out.append(g.get_blocks())
        g.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


# enough items for the multiple: pencils x block ids / pencils of an item >= 16 per SM
@pytest.mark.parametrize("n, nv, order", [
    ((5, 96, 32), (64, 32, 32), "xyz"), ((10, 48, 32), (64, 32, 32), "xyz"), ((11, 48, 32), (64, 32, 32), "xyz"),
    ((22, 32, 24), (64, 32, 32), "xyz"), ((23, 32, 24), (64, 32, 32), "xyz"), ((742, 5, 4), (16, 16, 16), "yxz"),
    ((743, 5, 4), (16, 16, 16), "yxz")])
def test_tables_of_48_kib(n, nv, order):
    code = f"import sys; sys.path[:0] = [{ROOT!r}, {os.path.dirname(os.path.abspath(__file__))!r}]\n" \
           f"import test_gpu_pass_smem as t; t.run({n}, {nv}, {order!r})"
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
