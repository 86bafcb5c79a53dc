"""P2G over cell-ordered particles and G2P through shared memory against float64:
particles at, on and beyond every wall, on cell faces and centres, in cell order and
shuffled, a count that ends inside a warp, and one non-finite particle, which reaches
its own 27 nodes per component and no other."""
import numpy as np
import pytest
import torch

from paper_2503_00868_gb300 import fluidstep as F

pytestmark = pytest.mark.gpu

NX, NY, NZ, DX = 21, 14, 17, 0.125


def particles(n, seed, order):
    rng = np.random.default_rng(seed)
    box = np.array([NX, NY, NZ]) * DX
    x = rng.uniform(-2.2 * DX, box + 2.2 * DX, (n, 3))
    snap = rng.random(n) < 0.2  # on faces and centres
    x[snap] = np.round(x[snap] / DX * 2) / 2 * DX
    if order == "cells":
        c = np.floor(x / DX)
        x = x[np.lexsort((c[:, 0], c[:, 1], c[:, 2]))]
    f = lambda *s: rng.standard_normal(s).astype(np.float32)  # noqa: E731
    return x.astype(np.float32), f(n, 3), f(n, 9), rng.uniform(0.5, 1.5, n).astype(np.float32)


def walk(x, comp):
    """(index, weight, offset) of the 27 nodes, in float64 from the float32 positions."""
    dims = np.array([NX + (comp == 0), NY + (comp == 1), NZ + (comp == 2)])
    sc = x.astype(np.float64) / DX - np.where(np.arange(3) == comp, 0.0, 0.5)
    base = np.floor(sc - 0.5)
    f = sc - base
    w = np.stack([0.5 * (1.5 - f) ** 2, 0.75 - (f - 1) ** 2, 0.5 * (f - 0.5) ** 2])
    for k in range(27):
        o = np.array([k % 3, (k // 3) % 3, k // 9])
        idx = (base + o).astype(int)
        ok = np.all((idx >= 0) & (idx < dims), axis=1)
        wt = w[o[0], :, 0] * w[o[1], :, 1] * w[o[2], :, 2]
        d = (idx + np.where(np.arange(3) == comp, 0.0, 0.5)) * DX - x
        yield idx, wt, d, ok


@pytest.mark.parametrize("order", ["cells", "shuffled"])
@pytest.mark.parametrize("n", [65536, 70001])
def test_transfers(order, n):
    x, v, C, m = particles(n, n, order)
    v[n // 2] = np.nan
    g = F.Grid(NX, NY, NZ, dx=DX)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    u, mass = g.zeros(), g.zeros()
    for _ in range(2):  # the second pass finds the workspace of the first
        F.fs_p2g(g.ctx, dev(x), dev(v), dev(C), dev(m), u, mass)
    got, gm = g.unpack(u), g.unpack(mass)
    dense = []
    for comp in range(3):
        shape = got[comp].shape
        mv, ms, mx = np.zeros(shape), np.zeros(shape), np.zeros(shape)
        for idx, wt, d, ok in walk(x, comp):
            val = v[:, comp] + (C[:, 3 * comp:3 * comp + 3] * d).sum(1)
            at = (idx[ok, 2], idx[ok, 1], idx[ok, 0])
            np.add.at(mv, at, (wt * m * val)[ok])
            np.add.at(ms, at, (wt * m)[ok])
            np.maximum.at(mx, at, np.where(np.isnan(val), 0.0, np.abs(val))[ok])
        want = np.where(ms > 0, mv / np.where(ms > 0, ms, 1), 0.0)
        assert np.array_equal(np.isnan(got[comp]), np.isnan(want))
        fine = ~np.isnan(want)
        # a node sums about n / cells * 27 products; each weight and product rounds a few units of 2^-24,
        # and a weight's factor near zero keeps an absolute error of the same size
        terms = 27 * n / (NX * NY * NZ)
        assert np.abs(gm[comp] - ms).max() <= (terms + 30) * 2.0 ** -24 * ms.max()
        heavy = fine & (ms > 1e-3 * ms.max())
        assert (np.abs(got[comp] - want)[heavy] <= (terms + 30) * 2.0 ** -24 * mx[heavy] * 1e3).all()
        dense.append(np.where(fine, want, 0.0).astype(np.float32))
    field = g.pack(dense)
    vo, Co = torch.empty(n, 3, device="cuda"), torch.empty(n, 9, device="cuda")
    F.fs_g2p(g.ctx, dev(x), vo, Co, field)
    for comp in range(3):
        wv, wC, big = np.zeros(n), np.zeros((n, 3)), np.abs(dense[comp]).max()
        for idx, wt, d, ok in walk(x, comp):
            val = np.zeros(n)
            val[ok] = dense[comp][idx[ok, 2], idx[ok, 1], idx[ok, 0]]
            wv += wt * val
            wC += (4 / DX ** 2) * (wt * val)[:, None] * d
        assert np.abs(vo[:, comp].cpu().numpy() - wv).max() <= 64 * 2.0 ** -24 * big
        assert np.abs(Co[:, 3 * comp:3 * comp + 3].cpu().numpy() - wC).max() <= 4 / DX ** 2 * 2 * DX * 64 * 2.0 ** -24 * big
