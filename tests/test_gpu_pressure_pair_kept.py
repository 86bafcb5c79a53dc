"""The last projection's pressure pair outlives calls that solve nothing."""
import pytest
import torch

from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["pbd_project", "p2g"])
def test_refined_pair_is_kept(call):
    n = 64
    g = F.Grid(n, n, n, dx=1.0 / n, tol_p=1e-7, maxit_p=20000, precond=F.FS_PRECOND_MG)
    g.set_mask(W.ellipsoid_blob(n, n, n, 0)[0])
    rc, st = g.project(g.pack(W.blurred_noise_mac(n, n, n, 3)))
    assert rc == F.FS_OK and st["restarts_p"] > 0  # the pressure is a pair of two terms
    before = [g.empty_cell(), g.empty_cell()]
    F.fs_pressure_pair(g.ctx, *before)
    assert all(bool(t.any()) for t in before)
    if call == "pbd_project":
        F.fs_pbd_project(g.ctx, g.pack(W.random_mac(n, n, n, 4)), True, 10, 0.5 * n * n)
    else:
        k = 1 << 17
        x = torch.rand(k, 3, device="cuda")
        F.fs_p2g(g.ctx, x, x - 0.5, torch.zeros(k, 9, device="cuda"), torch.ones(k, device="cuda"), g.zeros())
    after = [g.empty_cell(), g.empty_cell()]
    F.fs_pressure_pair(g.ctx, *after)
    assert all(torch.equal(a, b) for a, b in zip(before, after))
