"""P2G over cell-ordered particles on, and one or two float32 steps beside, the faces and
centres of cells whose size is not a power of two: the passes that order the particles
and the one that walks them have to agree on every particle's cell."""
import numpy as np
import pytest
import torch

from paper_2503_00868_gb300 import fluidstep as F

pytestmark = pytest.mark.gpu


def positions(n, dims, dx, seed):
    rng = np.random.default_rng(seed)
    half = rng.integers(-4, 2 * np.array(dims) + 5, (n, 3))  # halves of a cell, from two cells off the grid
    x = (half * np.float32(0.5 * dx)).astype(np.float32)
    for _ in range(2):
        x = np.where(rng.random((n, 3)) < 0.3, np.nextafter(x, np.float32(rng.choice([-9, 9])), dtype=np.float32), x)
    return x.astype(np.float32)


@pytest.mark.parametrize("dims,inv", [((75, 14, 17), 75.0), ((21, 50, 12), 49.0), ((13, 12, 60), 0.3)])
@pytest.mark.parametrize("order", ["cells", "shuffled"])
def test_mass_and_momentum(dims, inv, order):
    n, dx = 70000, 1.0 / inv
    x = positions(n, dims, dx, 3)
    if order == "cells":
        c = np.floor(x / dx)
        x = x[np.lexsort((c[:, 0], c[:, 1], c[:, 2]))]
    rng = np.random.default_rng(4)
    v = rng.standard_normal((n, 3)).astype(np.float32)
    m = rng.uniform(0.5, 1.5, n).astype(np.float32)
    g = F.Grid(*dims, dx=dx)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    u, mass = g.zeros(), g.zeros()
    F.fs_p2g(g.ctx, dev(x), dev(v), torch.zeros(n, 9, device="cuda"), dev(m), u, mass)
    got, gm = g.unpack(u), g.unpack(mass)
    f32dx = float(np.float32(dx))
    for comp in range(3):
        size = np.array(dims) + (np.arange(3) == comp)
        ms, mv, count = np.zeros(size[::-1]), np.zeros(size[::-1]), np.zeros(size[::-1])
        sc = x.astype(np.float64) / f32dx - np.where(np.arange(3) == comp, 0.0, 0.5)
        base = np.floor(sc - 0.5)
        f = sc - base
        w = np.stack([0.5 * (1.5 - f) ** 2, 0.75 - (f - 1) ** 2, 0.5 * (f - 0.5) ** 2])
        for k in range(27):
            o = np.array([k % 3, (k // 3) % 3, k // 9])
            idx = (base + o).astype(int)
            ok = np.all((idx >= 0) & (idx < size), axis=1)
            wt = w[o[0], :, 0] * w[o[1], :, 1] * w[o[2], :, 2] * m
            at = (idx[ok, 2], idx[ok, 1], idx[ok, 0])
            np.add.at(ms, at, wt[ok])
            np.add.at(mv, at, (wt * v[:, comp])[ok])
            np.add.at(count, at, m[ok])
        # a coordinate of up to max(dims) + 2 cells rounds twice (1 / dx, the product): a weight, of slope at most
        # 1, is off by that on each axis; the products and sums round as many times as there are terms
        per_term = 3 * 2 * (max(dims) + 2) * 2.0 ** -24 + 8 * 2.0 ** -24
        bound = count * (per_term + count.max() * 2.0 ** -24) + 1e-30
        assert (np.abs(gm[comp] - ms) <= bound).all()
        big = np.abs(v[:, comp]).max()
        assert (np.abs(got[comp] * gm[comp] - mv) <= 2 * big * bound + 1e-6 * np.abs(mv)).all()
