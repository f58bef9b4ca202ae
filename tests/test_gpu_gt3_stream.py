"""The plane-batched GT3 kernel's staging warps run ahead of the sweeping warps across
batches and items.  Streams as short as they can be (one to four planes: two or three
batches per item), more items than CTAs, tiles of one cell and tiles that wrap: bit for bit
the row-segment kernel's state (the same arithmetic, Section 3's tile + halo), in FP32 and
in 16-bit storage, dense and sparse."""
import numpy as np
import pytest

from paper_2504_21450_gb300 import inputs, vlasov

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    vlasov.load(build_if_missing=True)


@pytest.mark.parametrize("storage", [vlasov.VL_STORE_F32, vlasov.VL_STORE_BF16_SCALED])
@pytest.mark.parametrize("density", [1.0, 0.3])
@pytest.mark.parametrize("order", ["xyz", "yxz"])
@pytest.mark.parametrize("n", [(16, 16, 1), (17, 5, 2), (5, 33, 3), (22, 21, 4), (1, 1, 1)])
def test_short_streams_and_many_items(n, order, density, storage):
    nv = (16, 16, 16)  # 64 block ids x 4 chunks: more items than there are SMs
    init = inputs.random_blocks(n, nv, density, seed=101)
    out = []
    for kernel in (1, 2):
        g = vlasov.Grid(n, nv, (-8.0,) * 3, (1.0,) * 3, threshold=0.3, storage=storage)
        g.set_blocks(init.off, init.ids, init.vals)
        g.translate(0.1, order, 2, vlasov.VL_FORM_FUSED, check=True, kernel=kernel,
                    tile_rows=0 if kernel == 1 else 16)
        assert g.stats().kernel_used == kernel
        out.append(g.get_blocks())
        g.close()
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)
