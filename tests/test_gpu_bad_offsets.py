"""Offsets that are not a list's, alternating between nothing and everything, so that every
second cell claims all of the blocks: the call is refused in the time of a valid one, and does
not walk each claimed list first (131 thousand million ids here)."""
import time

import pytest

from paper_2504_21450_gb300 import vlasov

pytestmark = pytest.mark.gpu


def test_alternating_offsets():
    import torch
    vlasov.load(build_if_missing=True)
    n, m = (64, 32, 32), 1 << 22
    g = vlasov.Grid(n, (32, 32, 32), (-16.0,) * 3, (1.0,) * 3)
    cells = 64 * 32 * 32
    good = torch.arange(cells + 1, dtype=torch.int64, device="cuda") * (m // cells)
    ids = (torch.arange(m, device="cuda") % (m // cells)).to(torch.int16)
    vals = torch.ones((m, 64), dtype=torch.float32, device="cuda")
    bad = (torch.arange(cells + 1, device="cuda") % 2) * m
    bad[cells] = m
    for off in (good, bad, good, bad):
        torch.cuda.synchronize()
        t = time.perf_counter()
        if off is good:
            vlasov.vl_set_blocks(g.handle, m, off.data_ptr(), ids.data_ptr(), vals.data_ptr(), 1)
        else:
            with pytest.raises(vlasov.VlError) as e:
                vlasov.vl_set_blocks(g.handle, m, off.data_ptr(), ids.data_ptr(), vals.data_ptr(), 1)
            assert e.value.status == vlasov.VL_EINVAL
            # a valid call takes a few milliseconds, the walk would take seconds
            assert time.perf_counter() - t < 0.5
    g.close()
