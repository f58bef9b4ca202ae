"""vl_moments of grids with different velocity meshes, each used by a host thread of its own: the
kernel's shared memory differs (96 KiB and 48 KiB per CTA), the limit being a property of the
kernel and not of the grid, and no call is refused or changes its result.  Small grids, so
that the calls are short and the threads' launches often meet."""
import threading

import numpy as np
import pytest

from paper_2504_21450_gb300 import inputs, vlasov

pytestmark = pytest.mark.gpu


# 46 and 22 block ids; 512 and 128, split over CTAs, whose marginals a second kernel joins
@pytest.mark.parametrize("meshes", [((184, 4, 4), (88, 4, 4)), ((128, 32, 8), (64, 16, 8))])
def test_two_meshes_on_threads(meshes):
    import torch
    vlasov.load(build_if_missing=True)
    cases, failed = [], []
    for nv in meshes * 2:
        init = inputs.random_blocks((9, 2, 1), nv, 0.3, seed=111)
        with torch.cuda.stream(torch.cuda.Stream()):
            g = vlasov.Grid((9, 2, 1), nv, tuple(-0.5 * a for a in nv), (1.0,) * 3)
        g.set_blocks(init.off, init.ids, init.vals)
        cases.append((g, g.moments(), torch.zeros((18, 7), dtype=torch.float64, device="cuda")))
    torch.cuda.synchronize()

    def work(g, want, out):
        try:
            for i in range(3000):
                vlasov.vl_moments(g.handle, out.data_ptr(), 1)
            np.testing.assert_array_equal(out.cpu().numpy(), want)
        except Exception as e:  # reported by the main thread
            failed.append(e)

    threads = [threading.Thread(target=work, args=c) for c in cases]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for g, _, _ in cases:
        g.close()
    assert not failed, failed
