"""The recurrent pressure solver and its weight gradient with liquid along the first rows
of the first plane, whose 27 taps reach farthest before the cells, and along the last."""
import numpy as np
import pytest

import oracle as O
from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import workloads as W

pytestmark = pytest.mark.gpu

K = 3


def mask(nx, ny, nz, where):
    types = np.zeros((nz, ny, nx), np.uint8)
    if where == "first":
        types[0, 0] = 1
    elif where == "second":
        types[0, 1] = 1
    elif where == "last":
        types[-1, -1] = 1
    else:  # everything but one column of air
        types[:] = 1
        types[:, -1, nx // 2] = 0
    return types


@pytest.mark.parametrize("where", ["first", "second", "last", "most"])
@pytest.mark.parametrize("nx,ny,nz", [(4, 3, 2), (31, 6, 5), (32, 5, 7)])
def test_edge_rows(nx, ny, nz, where):
    types = mask(nx, ny, nz, where)
    w = np.random.default_rng(1).uniform(-0.004, 0.01, 27)
    w = 0.5 * (w + w[::-1])
    w[13] = 1.0 / 6.0
    w = w.astype(np.float32).astype(np.float64)
    g = F.Grid(nx, ny, nz, dx=1.0, pressure_solver=F.FS_SOLVER_PERCNN)
    F.fs_percnn_load(g.ctx, w, K)
    g.set_mask(types)
    liq = types == 1
    u = W.random_mac(nx, ny, nz, 3)
    b = -sum(np.diff(a, axis=2 - c) for c, a in enumerate(u)) * liq
    q = g.empty_cell()
    g.project(g.pack(u), q)
    d = sum(np.roll(np.pad(types != 2, 1), s, a)[1:-1, 1:-1, 1:-1].astype(float) for a in range(3) for s in (1, -1))
    p = np.zeros(types.shape)
    k3 = w.reshape(3, 3, 3)
    for _ in range(K):
        pp = np.pad(p, 1)
        nb = sum(np.roll(pp, s, a)[1:-1, 1:-1, 1:-1] for a in range(3) for s in (1, -1))
        r = np.pad((b - (d * p - nb)) * liq, 1)
        p = p + liq * sum(k3[z, y, x] * r[z:z + nz, y:y + ny, x:x + nx]
                          for z in range(3) for y in range(3) for x in range(3))
    # K sub-steps of 34 products and sums in FP32; the sub-steps contract
    assert np.linalg.norm(g.unpack_cell(q) - p) <= 34 * K * 2.0 ** -24 * np.linalg.norm(p)

    og = O.Grid(types, 1.0, 1 / 30, 0.0)
    O.set_percnn(og, w, K)
    q64 = np.where(liq, np.random.default_rng(7).standard_normal(types.shape), 0.0)
    b64 = O.poisson_apply(og, q64)
    lo, dwo = O.percnn_loss_grad(og, w, K, b64, q64)
    lg, dwg = F.fs_percnn_grad(g.ctx, g.pack_cell(b64), g.pack_cell(q64))
    # e = p - q is known to eps |q| in the energy norm, so the loss |e|^2 / |q|^2 to 2 sqrt(loss) eps + eps^2,
    # and the gradient, linear in e, to eps / sqrt(loss) and its own FP32 products and sums
    eps = 34 * K * 2.0 ** -24
    assert abs(lg - lo) <= 2 * np.sqrt(lo) * eps + eps ** 2 + 1e-6 * lo
    assert np.linalg.norm(dwg - dwo) <= (2 * eps / np.sqrt(lo) + 2e-3) * np.linalg.norm(dwo)
