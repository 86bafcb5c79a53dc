"""The multigrid's list kernels where a quad's neighbours in a row are not listed:
scattered masks, against the float64 V-cycle and, for the face volumes, against the
Jacobi-preconditioned solve; and a level whose restriction takes a thread per pair."""
import numpy as np
import pytest
import torch

from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import workloads as W

from test_gpu_mg_levels import COARSE_CELLS, coarsen, stored, vcycle

pytestmark = pytest.mark.gpu


def scatter(nx, ny, nz, liquid, solid):
    x = np.random.default_rng(11).random((nz, ny, nx))
    return np.where(x < liquid, 1, np.where(x < liquid + solid, 2, 0)).astype(np.uint8)


@pytest.mark.parametrize("nx,ny,nz,liquid,solid", [
    (45, 38, 41, 0.05, 0.30),    # mostly lone quads
    (64, 61, 67, 0.30, 0.30),    # broken rows, x a multiple of 4
    (133, 101, 92, 0.60, 0.10),
    (205, 190, 196, 1.0, 0.0),   # a thread per pair below level 0
])
def test_vcycle_rows_match_float64(nx, ny, nz, liquid, solid):
    types = scatter(nx, ny, nz, liquid, solid)
    levels = [types]
    while stored(levels[-1].shape, len(levels) == 1) > COARSE_CELLS:
        levels.append(coarsen(levels[-1]))
    r = np.random.default_rng(5).standard_normal(types.shape).astype(np.float32) * (types == 1)
    want = vcycle(levels, 0, r.astype(np.float64))
    g = F.Grid(nx, ny, nz, dx=1.0 / ny, precond=F.FS_PRECOND_MG)
    g.set_mask(types)
    z = g.empty_cell()
    for _ in range(2):
        g.precond_apply(g.pack_cell(r), z)
        got = g.unpack_cell(z)
        # each of the cycle's steps (at most 6 per level and 30 on the coarsest) rounds its result by a
        # few units of 2^-24; the sweeps do not amplify
        assert np.linalg.norm(got - want) <= 100 * 2.0 ** -24 * np.linalg.norm(want)
        assert np.all(got[types != 1] == 0.0)


@pytest.mark.parametrize("nx,ny,nz,liquid", [(45, 38, 41, 0.05), (64, 61, 67, 0.30), (133, 101, 92, 0.60)])
def test_viscosity_rows_match_jacobi(nx, ny, nz, liquid):
    types = scatter(nx, ny, nz, liquid, 0.0)
    dx, dt, tol = 1.0 / ny, 0.01, 1e-6
    u0 = W.blurred_noise_mac(nx, ny, nz, 3)
    out = []
    for precond in (F.FS_PRECOND_MG, F.FS_PRECOND_JACOBI):
        # nu dt / dx^2 = 2: the operator's eigenvalues lie in [1, 25]
        g = F.Grid(nx, ny, nz, dx=dx, dt=dt, nu=2.0 * dx * dx / dt, precond=precond, tol_p=1e-4, tol_v=tol)
        g.set_mask(types)
        u, v = g.zeros(), g.zeros()
        g.step(g.pack(u0), u, v)
        out.append(np.concatenate([a.ravel() for a in g.unpack(v)]))
    # a residual of tol leaves each solution within tol times the condition number
    assert np.linalg.norm(out[0] - out[1]) <= 2 * 25 * tol * np.linalg.norm(out[1])
