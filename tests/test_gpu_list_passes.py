"""The list passes of the constrained projection and the recurrent pressure solver
against plain float64 on dense arrays: rows that end inside a quad, single columns of
liquid, liquid at every wall, and a second mask on one context (whose vectors hold
values of the first off the new liquid)."""
import numpy as np
import pytest

from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import train_percnn as TP
from paper_2503_00868_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def masks(nx, ny, nz):
    rng = np.random.default_rng(nx)
    sparse = (rng.random((nz, ny, nx)) < 0.3).astype(np.uint8)
    sparse[rng.random(sparse.shape) < 0.1] = 2
    return [W.ellipsoid_blob(nx, ny, nz, 1)[0], sparse, W.all_liquid(nx, ny, nz)]


def faces(types):
    """Per component: free-to-move classes (fluid, surface) and the slices of the low and high cell."""
    p = np.pad(types, 1, constant_values=2)
    out = []
    for c in range(3):
        ax = 2 - c
        inner = [slice(1, -1)] * 3
        inner[ax] = slice(None)
        t = np.moveaxis(p[tuple(inner)], ax, 0)
        lo, hi = np.moveaxis(t[:-1], 0, ax), np.moveaxis(t[1:], 0, ax)
        fluid = (lo != 2) & (hi != 2) & ((lo == 1) | (hi == 1))
        out.append((fluid, fluid & (lo != hi)))
    return out


def diff(a, ax):
    return np.diff(a, axis=ax)


@pytest.mark.parametrize("nx,ny,nz", [(5, 4, 3), (31, 6, 9), (32, 17, 8), (70, 33, 20)])
@pytest.mark.parametrize("hold", [True, False])
def test_constrained_projection(nx, ny, nz, hold):
    g = F.Grid(nx, ny, nz, dx=0.5)
    iters, eps, dx = 25, 0.7, 0.5
    for types in masks(nx, ny, nz):
        g.set_mask(types)
        liq = types == 1
        u = [a.copy() for a in W.random_mac(nx, ny, nz, 3)]
        m = g.pack(u)
        norm = F.fs_pbd_project(g.ctx, m, hold, iters, eps)
        free = [f & ~s if hold else f for f, s in faces(types)]
        n = sum(np.take(f, range(f.shape[2 - c] - 1), 2 - c).astype(float)
                + np.take(f, range(1, f.shape[2 - c]), 2 - c) for c, f in enumerate(free))
        start = max(np.abs(a).max() for a in u)
        for _ in range(iters):
            C = sum(diff(a, 2 - c) for c, a in enumerate(u)) / dx * liq
            lam = np.where(liq, -C / (n / dx ** 2 + eps), 0.0)
            for c in range(3):
                pad = [(0, 0)] * 3
                pad[2 - c] = (1, 1)
                u[c] = u[c] - np.where(free[c], diff(np.pad(lam, pad), 2 - c), 0.0) / dx
        C = sum(diff(a, 2 - c) for c, a in enumerate(u)) / dx * liq
        # one rounding of the field, and per iteration one of Lambda (at most iters times the field's scale
        # times dx, moved by 1/dx)
        for got, want in zip(g.unpack(m), u):
            assert np.abs(got - want).max() <= 4 * iters * 2.0 ** -24 * start
        assert abs(norm - np.linalg.norm(C)) <= 1e-4 * np.linalg.norm(C) + 1e-5 * start * np.sqrt(liq.sum())


@pytest.mark.parametrize("nx,ny,nz,K", [(5, 4, 3, 4), (31, 6, 9, 7), (33, 18, 12, 12)])
def test_recurrent_solver(nx, ny, nz, K):
    g = F.Grid(nx, ny, nz, dx=1.0, pressure_solver=F.FS_SOLVER_PERCNN)
    w = np.asarray(TP.default_kernel(), np.float32).astype(np.float64).reshape(3, 3, 3)
    w = 0.5 * (w + w[::-1, ::-1, ::-1])
    F.fs_percnn_load(g.ctx, w, K)
    for types in masks(nx, ny, nz)[:2]:
        g.set_mask(types)
        liq = types == 1
        u = g.pack(W.random_mac(nx, ny, nz, 3))
        b = -sum(diff(a, 2 - c) for c, a in enumerate(W.random_mac(nx, ny, nz, 3))) * liq
        q = g.empty_cell()
        g.project(u, q)
        d = sum(np.roll(np.pad(types != 2, 1), s, a)[1:-1, 1:-1, 1:-1].astype(float) for a in range(3) for s in (1, -1))
        p = np.zeros(types.shape)
        for _ in range(K):
            pp = np.pad(p, 1)
            nb = sum(np.roll(pp, s, a)[1:-1, 1:-1, 1:-1] for a in range(3) for s in (1, -1))
            r = np.pad((b - (d * p - nb)) * liq, 1)
            p = p + liq * sum(w[z, y, x] * r[z:z + nz, y:y + ny, x:x + nx]
                              for z in range(3) for y in range(3) for x in range(3))
        # K sub-steps of 34 products and sums in FP32; the sub-steps contract
        assert np.linalg.norm(g.unpack_cell(q) - p) <= 34 * K * 2.0 ** -24 * np.linalg.norm(p)
