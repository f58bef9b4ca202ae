"""The allocation-free step wants no keep flags, whatever the values it writes: without the
limiter a plateau near the largest FP32 number overshoots to +infinity at its two edges, which
passes even the threshold of +infinity that this entry point has.  Row-segment kernel (an order
that ends in x, blocks across v = 0, an output that is only 4-byte aligned) and plane-batched
kernel.

The plateau's overshoot is at least 2 % of it (unlimited PPM next to a step, any Courant number
of the case), its top 0.08 % below the largest number, so both edge cells of every line along
the last axis overflow; the other two axes are constant, which the sweeps keep."""
import ctypes

import numpy as np
import pytest

from paper_2504_21450_gb300 import vlasov

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order, vmin, misaligned", [
    ("yzx", (-4.0, -4.0, -8.0), 0), ("xyz", (-3.0, -4.0, -8.0), 0), ("zxy", (-4.0, -3.0, -7.0), 0),
    ("xyz", (-4.0, -4.0, -8.0), 1), ("xyz", (-4.0, -4.0, -8.0), 0)])
def test_overflowing_values(order, vmin, misaligned):
    import torch
    vlasov.load(build_if_missing=True)
    n, nv, dt = (20, 18, 17), (8, 8, 16), 0.1
    axis = 2 - "xyz".index(order[2])  # of the cells as [z][y][x]
    cells = torch.ones(n[::-1], device="cuda")
    cells.narrow(axis, 5, 5).fill_(3.4e38)
    f = cells.reshape(1, -1, 1).expand(16 * 4, -1, 16).contiguous()
    space = vlasov.vl_space_desc((ctypes.c_int * 3)(*n), (ctypes.c_double * 3)(1, 1, 1), (ctypes.c_double * 3)(0, 0, 0))
    vm = vlasov.vl_vmesh_desc((ctypes.c_int * 3)(*nv), (ctypes.c_double * 3)(*vmin),
                              (ctypes.c_double * 3)(1, 1, 1), (ctypes.c_int * 3)(4, 4, 4))
    room = torch.zeros(f.numel() + 4, device="cuda")
    out = room[misaligned:misaligned + f.numel()]
    mass = torch.zeros(1, dtype=torch.float64, device="cuda")
    st = vlasov.vl_translate_dense_noalloc(space, vm, dt, order, 0, f.data_ptr(), out.data_ptr(), mass.data_ptr(),
                                           torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert st == vlasov.VL_OK, vlasov.status_str(st)
    got = out.reshape(64, *n[::-1], 16).cpu().numpy()
    inf = np.isposinf(got)
    assert np.all(inf.sum(axis=axis + 1) == 2)
    assert np.all(np.isfinite(got) | inf)
    assert not room[:misaligned].any() and not room[misaligned + f.numel():].any()
