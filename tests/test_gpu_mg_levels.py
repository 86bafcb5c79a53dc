"""The multigrid V-cycle against a plain float64 V-cycle on dense arrays, at sizes
that take each way through its levels: a level 0 that is its own coarsest one, all
levels below level 0 in one block, tile kernels with remainders on every axis (and
both tile heights), and a level that takes one launch per step."""
import numpy as np
import pytest
import torch

from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import workloads as W

pytestmark = pytest.mark.gpu

OMEGA, COARSE_SWEEPS, COARSE_CELLS = 0.8, 30, 3072


def shifts(a):
    p = np.pad(a, 1)
    return (p[1:-1, 1:-1, :-2] + p[1:-1, 1:-1, 2:] + p[1:-1, :-2, 1:-1] + p[1:-1, 2:, 1:-1] + p[:-2, 1:-1, 1:-1]
            + p[2:, 1:-1, 1:-1])


def coarsen(types):
    """Air where any child is air, else liquid where any is liquid, else solid (off the grid: solid)."""
    pad = [(0, n % 2) for n in types.shape]
    t = np.pad(types, pad, constant_values=2)
    c = t.reshape(t.shape[0] // 2, 2, t.shape[1] // 2, 2, t.shape[2] // 2, 2)
    air, liq = (c == 0).any(axis=(1, 3, 5)), (c == 1).any(axis=(1, 3, 5))
    return np.where(air, 0, np.where(liq, 1, 2)).astype(np.uint8)


def stored(shape, level0):
    """Elements of a level's stored array, which decide where the hierarchy ends."""
    nz, ny, nx = shape
    if level0:
        return (nx + 4) // 4 * 4 * (ny + 1) * (nz + 3)
    return (nx + 8) // 4 * 4 * (ny + 2) * (nz + 2)


def axis_prolong(c, n, axis):
    """Cell-centred linear interpolation along one axis, zero off the grid."""
    c = np.moveaxis(c, axis, 0)
    p = np.pad(c, [(1, 1)] + [(0, 0)] * (c.ndim - 1))
    i = np.arange(n)
    out = 0.75 * p[i // 2 + 1] + 0.25 * p[np.where(i % 2 == 1, i // 2 + 2, i // 2)]
    return np.moveaxis(out, 0, axis)


def axis_restrict(f, nc, axis):
    """The transpose of axis_prolong."""
    f = np.moveaxis(f, axis, 0)
    out = np.zeros((nc + 2,) + f.shape[1:])
    i = np.arange(f.shape[0])
    np.add.at(out, i // 2 + 1, 0.75 * f)
    np.add.at(out, np.where(i % 2 == 1, i // 2 + 2, i // 2), 0.25 * f)
    return np.moveaxis(out[1:-1], 0, axis)


def vcycle(levels, l, r):
    types = levels[l]
    liq = types == 1
    d = shifts(((types == 1) | (types == 0)).astype(np.float64)) * liq
    sc = 0.25 ** l
    inv = np.where(d > 0, OMEGA / (sc * np.where(d > 0, d, 1.0)), 0.0) * liq
    resid = lambda e: (r - sc * (d * e - shifts(e))) * liq  # noqa: E731
    e = inv * r
    if l == len(levels) - 1:
        for _ in range(COARSE_SWEEPS - 1):
            e = e + inv * resid(e)
        return e
    e = e + inv * resid(e)
    f = resid(e)
    for axis in range(3):
        f = axis_restrict(f, levels[l + 1].shape[axis], axis)
    c = vcycle(levels, l + 1, f / 8.0 * (levels[l + 1] == 1))
    for axis in range(3):
        c = axis_prolong(c, types.shape[axis], axis)
    e = e + c * liq
    e = e + inv * resid(e)
    return e + inv * resid(e)


@pytest.mark.parametrize("nx,ny,nz,scene", [
    (9, 8, 7, "blob"),          # one level
    (17, 16, 20, "box"),        # closed: every level below in one block
    (33, 30, 29, "blob"),       # the same, odd at every level
    (70, 61, 67, "blob"),       # one level of 4 x 4 tiles
    (131, 66, 90, "spheres"),   # two levels of tiles, three ragged pieces along x
    (6, 200, 9, "blob"),        # a quad and a half per row
    (201, 178, 190, "blob"),    # level 1 by lists, then 8 x 8 tiles
])
def test_vcycle_matches_float64(nx, ny, nz, scene):
    types = {"blob": lambda: W.ellipsoid_blob(nx, ny, nz, 3)[0], "box": lambda: W.all_liquid(nx, ny, nz),
             "spheres": lambda: W.sphere_union(nx, ny, nz, 1, occ_range=(0.01, 0.9))[0]}[scene]()
    levels = [types]
    while stored(levels[-1].shape, len(levels) == 1) > COARSE_CELLS:
        levels.append(coarsen(levels[-1]))
    r = np.random.default_rng(5).standard_normal(types.shape).astype(np.float32) * (types == 1)
    want = vcycle(levels, 0, r.astype(np.float64))
    g = F.Grid(nx, ny, nz, dx=1.0 / ny, precond=F.FS_PRECOND_MG)
    g.set_mask(types)
    z = g.empty_cell()
    for _ in range(2):  # the second apply starts from the first one's work arrays
        g.precond_apply(g.pack_cell(r), z)
        got = g.unpack_cell(z)
        # each of the cycle's steps (at most 6 per level and 30 on the coarsest) rounds its result by a
        # few units of 2^-24; the sweeps do not amplify
        assert np.linalg.norm(got - want) <= 100 * 2.0 ** -24 * np.linalg.norm(want)
        assert np.all(got[types != 1] == 0.0)
