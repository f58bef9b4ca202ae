"""The allocation-free step through the plane-batched kernel: the bits of the regular entry
point on ragged and tiny grids; an output that is only 4-byte aligned keeps the row-segment
kernel and gives the same values."""
import ctypes

import numpy as np
import pytest

from paper_2504_21450_gb300 import inputs, vlasov

from test_zz_no_alloc import to_storage

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("misaligned", [0, 1])
@pytest.mark.parametrize("order, limiter", [("xyz", 1), ("zxy", 1), ("yxz", 0)])
@pytest.mark.parametrize("n", [(35, 20, 12), (5, 3, 2), (16, 17, 1)])
def test_same_bits_as_the_regular_entry_point(n, order, limiter, misaligned):
    import torch
    vlasov.load(build_if_missing=True)
    nv, vmin, dt = (8, 8, 16), (-4.0, -4.0, -8.0), 0.1
    nb, ncells = 16, int(np.prod(n))
    init = inputs.random_blocks(n, nv, 1.0, seed=78)
    g = vlasov.Grid(n, nv, vmin, (1.0,) * 3, threshold=0.0)
    g.set_blocks(init.off, init.ids, init.vals)
    g.translate(dt, order, 1, vlasov.VL_FORM_FUSED, limiter=bool(limiter), check=True)
    want, want_mass = to_storage(*g.get_blocks(), ncells, nb), g.stats().mass
    g.close()
    space = vlasov.vl_space_desc((ctypes.c_int * 3)(*n), (ctypes.c_double * 3)(1, 1, 1), (ctypes.c_double * 3)(0, 0, 0))
    vm = vlasov.vl_vmesh_desc((ctypes.c_int * 3)(*nv), (ctypes.c_double * 3)(*vmin),
                              (ctypes.c_double * 3)(1, 1, 1), (ctypes.c_int * 3)(4, 4, 4))
    f = torch.from_numpy(to_storage(init.off, init.ids, init.vals, ncells, nb)).cuda()
    room = torch.zeros(f.numel() + 4, device="cuda")
    out = room[misaligned:misaligned + f.numel()]
    mass = torch.zeros(1, dtype=torch.float64, device="cuda")
    st = vlasov.vl_translate_dense_noalloc(space, vm, dt, order, limiter, f.data_ptr(), out.data_ptr(),
                                           mass.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert st == vlasov.VL_OK, vlasov.status_str(st)
    got = out.cpu().numpy()
    if misaligned and order[2] != "z":  # the row-segment kernel's sign-generic window
        # both windows round a few times per value: a few units in the last place of max f
        np.testing.assert_allclose(got, want, rtol=0, atol=1e-5 * np.abs(want).max())
    else:
        np.testing.assert_array_equal(got, want)
    assert abs(float(mass.item()) - want_mass) <= 1e-6 * abs(want_mass)
    assert not room[:misaligned].any() and not room[misaligned + f.numel():].any()
