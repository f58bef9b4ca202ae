"""The plane-batched kernel's sweeping warps wait for the output slots of a sparse next layout,
however long the staging warps take to write them: with VLGT_FAULT=slow_slots those sleep for
50 us first, ten times as long as a batch is swept, and the state has the bits of the
row-segment kernel (the same arithmetic).  FP32 and 16-bit storage publish a batch through
different arrivals, and 16-bit storage stages rows in two ways (sweep 0 along x or not)."""
import numpy as np
import pytest

from paper_2504_21450_gb300 import inputs, vlasov

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [vlasov.VL_STORE_F32, vlasov.VL_STORE_BF16_SCALED, vlasov.VL_STORE_F16_SCALED])
@pytest.mark.parametrize("order", ["xyz", "yxz"])
@pytest.mark.parametrize("n", [(22, 21, 13), (17, 3, 2), (70, 18, 7)])
def test_slots_written_late(n, order, storage, monkeypatch):
    vlasov.load(build_if_missing=True)
    nv = (16, 16, 16)  # 64 block ids x 4 chunks: several items per CTA
    init = inputs.random_blocks(n, nv, 0.02, seed=107)
    out = []
    for kernel in (2, 1):
        g = vlasov.Grid(n, nv, (-8.0,) * 3, (1.0,) * 3, threshold=0.05, storage=storage)
        g.set_blocks(init.off, init.ids, init.vals)
        if kernel == 1:
            monkeypatch.setenv("VLGT_FAULT", "slow_slots")
        g.translate(0.1, order, 1, vlasov.VL_FORM_FUSED, check=True, kernel=kernel,
                    tile_rows=16 if kernel == 2 else 0)
        monkeypatch.delenv("VLGT_FAULT", raising=False)
        s = g.stats()
        assert s.kernel_used == kernel
        assert s.union_blocks < 0.9 * 64 * np.prod(n)  # the next layout is sparse
        out.append(g.get_blocks())
        g.close()
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)
