"""Per-cell lists in and out against the lists they came from: windows that wrap and cut
groups of eight cells, rows around 8 and 64 cells, block ids split over warps, host, page-
locked and device buffers, values that are only 4-byte aligned, 16-bit storage (a state read
back and set again stays as it is), lists of planes that are not in order, bad lists."""
import numpy as np
import pytest

from paper_2504_21450_gb300 import inputs, vlasov

pytestmark = pytest.mark.gpu
NV = (16, 8, 40)  # 80 block ids: more than one part where the cells are few


def window(init, n, origin, size):
    off, ids, vals = [0], [], []
    for z in range(size[2]):
        for y in range(size[1]):
            for x in range(size[0]):
                c = ((origin[0] + x) % n[0] + n[0] * ((origin[1] + y) % n[1]
                                                      + n[1] * ((origin[2] + z) % n[2])))
                s = slice(init.off[c], init.off[c + 1])
                ids.append(init.ids[s])
                vals.append(init.vals[s])
                off.append(off[-1] + ids[-1].size)
    return np.array(off), np.concatenate(ids), np.concatenate(vals)


def grid(n, storage=vlasov.VL_STORE_F32):
    vlasov.load(build_if_missing=True)
    return vlasov.Grid(n, NV, (-8.0, -4.0, -20.0), (1.0,) * 3, storage=storage)


@pytest.mark.parametrize("n, origin, size", [
    ((1, 1, 1), (0, 0, 0), (1, 1, 1)), ((9, 3, 2), (-2, 1, 1), (9, 2, 2)), ((7, 4, 3), (5, -1, 2), (3, 4, 1)),
    ((63, 2, 2), (60, 0, 0), (8, 2, 2)), ((70, 3, 2), (61, 2, 1), (13, 3, 2)), ((64, 5, 3), (0, 0, 1), (64, 5, 2))])
@pytest.mark.parametrize("density", [1.0, 0.25])
def test_windows(n, origin, size, density):
    init = inputs.random_blocks(n, NV, density, seed=104)
    g = grid(n)
    g.set_blocks(init.off, init.ids, init.vals)
    for a, b in zip(g.get_blocks(), (init.off, init.ids, init.vals)):
        np.testing.assert_array_equal(a, b)
    for a, b in zip(g.get_window(origin, size), window(init, n, origin, size)):
        np.testing.assert_array_equal(a, b)
    g.close()


@pytest.mark.parametrize("storage", [vlasov.VL_STORE_F32, vlasov.VL_STORE_BF16_SCALED, vlasov.VL_STORE_F16_SCALED])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("where", ["device", "page-locked"])
def test_buffers(where, shift, storage):
    """A state set from host lists, read into a buffer and set again from it."""
    import torch
    n = (37, 5, 3)
    init = inputs.random_blocks(n, NV, 0.4, seed=105)
    m = init.ids.size
    g, h = grid(n, storage), grid(n, storage)
    g.set_blocks(init.off, init.ids, init.vals)
    want = g.get_blocks()
    dev = where == "device"
    kw = {"device": "cuda"} if dev else {"pin_memory": True}
    off = torch.zeros(init.off.size, dtype=torch.int64, **kw)
    ids = torch.zeros(m, dtype=torch.int16, **kw)
    room = torch.zeros(64 * m + 8, dtype=torch.float32, **kw)
    vals = room[shift:shift + 64 * m]
    vlasov.vl_get_blocks(g.handle, m, off.data_ptr(), ids.data_ptr(), vals.data_ptr(), int(dev))
    torch.cuda.synchronize()
    np.testing.assert_array_equal(off.cpu().numpy(), want[0])
    np.testing.assert_array_equal(ids.cpu().numpy().view(np.uint16), want[1])
    np.testing.assert_array_equal(vals.cpu().numpy().reshape(m, 64), want[2])
    assert not room[:shift].any() and not room[shift + 64 * m:].any()
    vlasov.vl_set_blocks(h.handle, m, off.data_ptr(), ids.data_ptr(), vals.data_ptr(), int(dev))
    for a, b in zip(h.get_blocks(), want):
        np.testing.assert_array_equal(a, b)
    assert h.export() == g.export()
    g.close()
    h.close()


def test_planes_in_any_order_and_bad_lists():
    import torch
    n = (11, 3, 6)
    init = inputs.random_blocks(n, NV, 0.5, seed=106)
    g = grid(n)
    g.set_blocks(init.off, init.ids, init.vals)
    off, ids, vals = window(init, n, (0, 0, 4), (11, 3, 3))  # wraps
    rng = np.random.default_rng(7)
    new = rng.random(vals.shape).astype(np.float32)
    want = init.vals.copy()
    at = np.concatenate([np.arange(init.off[c], init.off[c + 1])
                         for z in (4, 5, 0) for c in range(33 * z, 33 * z + 33)])
    want[at] = new
    order = np.concatenate([rng.permutation(np.arange(off[c], off[c + 1])) for c in range(99)])
    for o in (np.arange(ids.size), order):  # ascending, then shuffled within the cells
        i, v = np.ascontiguousarray(ids[o]), np.ascontiguousarray(new[o])
        vlasov.vl_set_blocks_planes(g.handle, 4, 3, i.size, off.ctypes.data, i.ctypes.data, v.ctypes.data, 0)
        np.testing.assert_array_equal(g.get_blocks()[2], want)
        vlasov.vl_set_blocks_planes(g.handle, 4, 3, i.size, off.ctypes.data, ids.ctypes.data, vals.ctypes.data, 0)
        np.testing.assert_array_equal(g.get_blocks()[2], init.vals)
    dv = torch.from_numpy(init.vals).cuda()
    for bad_off, bad_ids in ((init.off[::-1].copy(), init.ids), (init.off + 1, init.ids),
                             (init.off, init.ids[::-1].copy()), (init.off, np.full_like(init.ids, 80))):
        do = torch.from_numpy(bad_off).cuda()
        di = torch.from_numpy(bad_ids.view(np.int16)).cuda()
        with pytest.raises(vlasov.VlError) as e:
            vlasov.vl_set_blocks(g.handle, init.ids.size, do.data_ptr(), di.data_ptr(),
                                 dv.data_ptr(), 1)
        assert e.value.status == vlasov.VL_EINVAL
    g.close()
