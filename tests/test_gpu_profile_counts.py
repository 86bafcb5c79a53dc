"""The profile counts what did work: with every iteration timed, an entry of a solve has
as many launches as the solve has iterations, though a batch enqueues more; the network's
flops are those of the cells that each layer must compute."""
import numpy as np
import pytest

from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import train_precond as T
from paper_2503_00868_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def network_flops(types):
    near, cells = types == 1, []
    for _ in range(5):  # within 0 .. 4 cells of the liquid
        cells.append(int(near.sum()))
        for ax in range(3):
            p = np.pad(near, [(1, 1) if a == ax else (0, 0) for a in range(3)])
            lo, hi = (np.take(p, range(s, s + types.shape[ax]), ax) for s in (0, 2))
            near = near | lo | hi
    return sum(54.0 * c * n for c, n in zip((2 * 16, 256, 256, 256, 16), cells[::-1]))


@pytest.mark.parametrize("role,precond", [("net", F.FS_PRECOND_LEARNED), ("net_mg", F.FS_PRECOND_LEARNED_MG)])
def test_network(role, precond):
    nx, ny, nz = 45, 38, 41
    types = W.sphere_union(nx, ny, nz, 2, occ_range=(0.02, 0.9))[0]
    g = F.Grid(nx, ny, nz, dx=1.0 / ny, tol_p=1e-5, precond=precond, maxit_p=2000, check_every=8)
    F.fs_net_load(g.ctx, T.role_weights(role))
    g.set_mask(types)
    g.profile(1)
    rc, st = g.project(g.pack(W.random_mac(nx, ny, nz, 5)))
    prof = g.profile_read()
    assert rc == F.FS_OK and st["iters_p"] % 8  # the last batch holds iterations after convergence
    launches, _, flops, every = prof["net_apply"]
    assert launches == every == st["iters_p"]
    assert flops / launches == network_flops(types)
    assert prof["fcg_vectors"][0] == st["iters_p"]


@pytest.mark.parametrize("precond", [F.FS_PRECOND_JACOBI, F.FS_PRECOND_MIC0, F.FS_PRECOND_MG])
def test_solves(precond):
    n = 40
    g = F.Grid(n, n, n, dx=1.0 / n, nu=0.01, tol_p=1e-5, tol_v=1e-6, precond=precond, maxit_p=2000, check_every=7)
    g.set_mask(W.ellipsoid_blob(n, n, n, 2)[0])
    for _ in range(2):  # batches of `check_every`, then by the last count
        g.profile(1)
        rc, st = g.step(g.pack(W.blurred_noise_mac(n, n, n, 3)), g.zeros())
        prof = g.profile_read()
        assert rc == F.FS_OK
        p = {F.FS_PRECOND_MIC0: "mic0_apply", F.FS_PRECOND_MG: "mg_vcycle_p"}.get(precond)
        for k in ["pressure_spmv", "pressure_update"] + ([p] if p else []):
            assert prof[k][0] == prof[k][3] == st["iters_p"], (k, prof[k], st)
        for k in ["visc_spmv", "visc_update"] + (["mg_vcycle_v"] if precond == F.FS_PRECOND_MG else []):
            assert prof[k][0] == prof[k][3] == st["iters_v"], (k, prof[k], st)
