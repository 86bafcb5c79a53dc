"""Flexible CG repeats bit for bit: every kernel of an iteration reads what the launch
before it wrote, whatever ran on the GPU before (the direction coefficients change
from iteration to iteration in one buffer)."""
import pytest
import torch

from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import train_precond as T
from paper_2503_00868_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("role,precond", [("net", F.FS_PRECOND_LEARNED), ("net_mg", F.FS_PRECOND_LEARNED_MG)])
def test_projection_repeats(role, precond):
    n = 40
    runs = []
    for busy in (0, 1, 0):
        g = F.Grid(n, n, n, dx=1.0 / n, tol_p=1e-6, precond=precond, maxit_p=2000)
        F.fs_net_load(g.ctx, T.role_weights(role))
        g.set_mask(W.sphere_union(n, n, n, 2)[0])
        u = g.pack(W.random_mac(n, n, n, 5))
        if busy:  # the GPU is still at work when the solve is enqueued
            a = torch.randn(4096, 4096, device="cuda")
            for _ in range(20):
                a = a @ a * 1e-3
        rc, st = g.project(u)
        assert rc == F.FS_OK and st["fallbacks"] == 0 and st["true_relres_p"] <= 1e-6
        runs.append((st["iters_p"], u))
    for it, u in runs[1:]:
        assert it == runs[0][0] and all(torch.equal(x, y) for x, y in zip(u, runs[0][1]))
