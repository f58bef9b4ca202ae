"""The plane-batched kernel's total mass, summed in FP32 with a compensation over all items of a
CTA, loses nothing when it is handed on in FP64.

dt = 0 leaves every value as it is.  The values are whole numbers below 2**20, so the eight
that a thread adds at a time have an exact FP32 sum, the compensated sum is exact (Fast2Sum:
its high part is never the smaller one once it rounds), and so are the FP64 sums of whole
numbers below 2**53 and the scaling by a power of two: the mass has to be the exact one.  A
thread's sum passes 2**24 after a few planes, from where its high part alone is short."""
import ctypes

import numpy as np
import pytest

from paper_2504_21450_gb300 import inputs, vlasov

from test_zz_no_alloc import to_storage

pytestmark = pytest.mark.gpu
NV, VMIN = (8, 8, 16), (-4.0, -4.0, -8.0)


def case(n):
    init = inputs.random_blocks(n, NV, 1.0, seed=108)
    rng = np.random.default_rng(109)
    return init, rng.integers(1, 2 ** 20, init.vals.shape).astype(np.float32)


@pytest.mark.parametrize("order", ["xyz", "zxy"])
@pytest.mark.parametrize("n", [(16, 16, 40), (35, 20, 33)])
def test_step(n, order):
    vlasov.load(build_if_missing=True)
    init, vals = case(n)
    g = vlasov.Grid(n, NV, VMIN, (1.0,) * 3)
    g.set_blocks(init.off, init.ids, vals)
    g.translate(0.0, order, 1, vlasov.VL_FORM_FUSED, check=True, kernel=1)
    np.testing.assert_array_equal(g.get_blocks()[2], vals)
    assert g.stats().mass == float(vals.astype(np.int64).sum())
    g.close()


@pytest.mark.parametrize("order", ["xyz", "zxy"])
@pytest.mark.parametrize("n", [(16, 16, 40), (35, 20, 33)])
def test_allocation_free_step(n, order):
    import torch
    vlasov.load(build_if_missing=True)
    init, vals = case(n)
    space = vlasov.vl_space_desc((ctypes.c_int * 3)(*n), (ctypes.c_double * 3)(1, 1, 1), (ctypes.c_double * 3)(0, 0, 0))
    vm = vlasov.vl_vmesh_desc((ctypes.c_int * 3)(*NV), (ctypes.c_double * 3)(*VMIN),
                              (ctypes.c_double * 3)(1, 1, 1), (ctypes.c_int * 3)(4, 4, 4))
    f = torch.from_numpy(to_storage(init.off, init.ids, vals, int(np.prod(n)), 16)).cuda()
    out, mass = torch.zeros_like(f), torch.zeros(1, dtype=torch.float64, device="cuda")
    st = vlasov.vl_translate_dense_noalloc(space, vm, 0.0, order, 1, f.data_ptr(), out.data_ptr(),
                                           mass.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert st == vlasov.VL_OK, vlasov.status_str(st)
    assert torch.equal(out, f)
    assert float(mass.item()) == float(vals.astype(np.int64).sum())
