"""Velocity moments and total mass against FP64 sums over the listed values, at the edges of
the kernel: groups of eight cells (rows shorter and longer than eight and 64 cells), runs
of blocks along vx, ids split over CTAs, sparse cells, 16-bit storage, values of any size,
infinities, and a mesh too wide for the marginals.

Tolerance: 2**-44 of the sum of magnitudes, far above the rounding of the FP64 sums; cells of
a few blocks, whose values span many decades, are held to that rounding itself."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2504_21450_gb300 import inputs, vlasov

pytestmark = pytest.mark.gpu
TOL = 2.0 ** -44


def reference(g, nv, vmin, dv):
    off, ids, vals = g.get_blocks()
    cell = np.repeat(np.arange(off.size - 1), np.diff(off))
    nb = [v // 4 for v in nv]
    b, l = ids.astype(np.int64), np.arange(64)
    bc = [b % nb[0], (b // nb[0]) % nb[1], b // (nb[0] * nb[1])]
    within = [l & 3, (l >> 2) & 3, l >> 4]
    v = [vmin[d] + (4 * bc[d][:, None] + within[d] + 0.5) * dv[d] for d in range(3)]
    f, n = vals.astype(np.float64), off.size - 1
    dv3 = dv[0] * dv[1] * dv[2]

    def total(w):
        return np.bincount(cell, weights=w.sum(axis=1), minlength=n)
    out, size = np.zeros((n, 7)), np.zeros((n, 7))
    out[:, 0], size[:, 0] = total(f), total(np.abs(f))
    for d in range(3):
        out[:, 1 + d], size[:, 1 + d] = total(f * v[d]), total(np.abs(f * v[d]))
        mean = out[:, 1 + d] / np.where(out[:, 0] != 0, out[:, 0], 1.0)
        w = (v[d] - mean[cell][:, None]) ** 2
        out[:, 4 + d], size[:, 4 + d] = total(f * w), total(np.abs(f) * w)
    return out * dv3, size * dv3


def check(n, nv, density, storage, scale=1.0, seed=102):
    vmin, dv = tuple(-0.4 * a for a in nv), (1.0, 0.5, 0.75)
    init = inputs.random_blocks(n, nv, density, seed=seed, scale=scale)
    g = vlasov.Grid(n, nv, vmin, dv, storage=storage)
    g.set_blocks(init.off, init.ids, init.vals)
    got, mass = g.moments(), g.mass()
    want, size = reference(g, nv, vmin, dv)
    g.close()
    assert np.all(np.abs(got - want) <= TOL * size)
    assert abs(mass - want[:, 0].sum()) <= TOL * size[:, 0].sum()


@pytest.mark.parametrize("storage", [vlasov.VL_STORE_F32, vlasov.VL_STORE_BF16_SCALED, vlasov.VL_STORE_F16_SCALED])
@pytest.mark.parametrize("n, nv, density", [
    ((1, 1, 1), (4, 4, 4), 1.0), ((9, 3, 2), (8, 8, 8), 0.2), ((7, 2, 3), (40, 8, 4), 0.7),
    ((70, 3, 2), (8, 12, 8), 0.5), ((3, 2, 2), (32, 32, 32), 0.3), ((64, 9, 5), (16, 4, 4), 1.0)])
def test_moments_and_mass(n, nv, density, storage):
    check(n, nv, density, storage)


@pytest.mark.parametrize("scale", [1e-41, 1e-20, 2e36, 3e38])
def test_values_of_any_size(scale):
    check((9, 3, 2), (16, 8, 8), 0.8, vlasov.VL_STORE_F32, scale)


def test_mesh_too_wide_for_the_marginals():
    check((3, 2, 1), (1600, 4, 8), 0.5, vlasov.VL_STORE_F32)


def test_infinities_stay_in_their_cell():
    n, nv = (9, 2, 1), (8, 8, 8)
    init = inputs.random_blocks(n, nv, 1.0, seed=103)
    vals = init.vals.copy()
    vals[3 * 8 + 2, 5] = np.inf   # block 2 of cell 3
    vals[5 * 8 + 1, 9] = np.nan   # block 1 of cell 5
    g = vlasov.Grid(n, nv, (-4.0,) * 3, (1.0,) * 3)
    g.set_blocks(init.off, init.ids, init.vals)
    clean, (_, size) = g.moments(), reference(g, nv, (-4.0,) * 3, (1.0,) * 3)
    g.set_blocks(init.off, init.ids, vals)
    got, mass = g.moments(), g.mass()
    g.close()
    assert got[3, 0] == np.inf and np.isinf(got[3, 1:4]).all() and np.isnan(got[3, 4:]).all()
    assert np.isnan(got[5]).all() and np.isnan(mass)
    other = np.delete(np.arange(18), [3, 5])
    assert np.all(np.abs(got - clean)[other] <= 2 * TOL * size[other])


@pytest.mark.parametrize("nv, storage", [((4, 4, 4), vlasov.VL_STORE_F32), ((8, 4, 8), vlasov.VL_STORE_F32),
                                         ((8, 8, 4), vlasov.VL_STORE_BF16_SCALED)])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e30])
def test_few_blocks_to_the_rounding_of_fp64(nv, storage, scale):
    """n and n V_d against exact rationals.  Bound: each value's share passes one rounding per
    block along an axis (at most 4 here), nv / 4 + 2 in the sum over a marginal, 3 for the
    product with v and dv^3: 16 * 2**-53 of the sum of magnitudes, and 2**-60 for the rest
    below the places."""
    n, vmin, dv = (9, 2, 1), (-1.5, -2.0, -0.75), (1.0, 0.5, 0.25)
    init = inputs.random_blocks(n, nv, 1.0, seed=104)
    r = np.random.Generator(np.random.PCG64(105))
    vals = (init.vals * np.exp(r.uniform(-30.0, 0.0, init.vals.shape)) * scale).astype(np.float32)
    g = vlasov.Grid(n, nv, vmin, dv, storage=storage)
    g.set_blocks(init.off, init.ids, vals)
    got, mass = g.moments(), g.mass()
    off, ids, vals = g.get_blocks()
    g.close()
    nb, dv3, total = [v // 4 for v in nv], Fraction(dv[0] * dv[1] * dv[2]), Fraction(0)
    for c in range(off.size - 1):
        want, size = [Fraction(0)] * 4, [Fraction(0)] * 4
        for b, block in zip(ids[off[c]:off[c + 1]].astype(int), vals[off[c]:off[c + 1]]):
            bc = (b % nb[0], b // nb[0] % nb[1], b // (nb[0] * nb[1]))
            for l in range(64):
                f = Fraction(float(block[l]))
                w = [Fraction(1)] + [Fraction(vmin[d]) + (4 * bc[d] + (l >> 2 * d & 3) + Fraction(1, 2)) * Fraction(dv[d])
                                     for d in range(3)]
                for m in range(4):
                    want[m] += f * w[m]
                    size[m] += abs(f * w[m])
        total += want[0] * dv3
        for m in range(4):
            assert abs(Fraction(float(got[c, m])) - want[m] * dv3) <= (16 * Fraction(2) ** -53 + Fraction(2) ** -60) * size[m] * dv3
    assert abs(Fraction(mass) - total) <= 16 * Fraction(2) ** -53 * total
