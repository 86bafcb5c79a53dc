"""Flexible CG over the list of active quads: after a change of mask on one context
(its vectors then hold values of the old mask off the new liquid) a projection meets
the oracle as on a new context, with the learned preconditioner in both roles and on
sizes whose rows end inside a quad; a closed box keeps its null mode out."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import train_precond as T
from paper_2503_00868_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("role", ["net", "net_mg"])
@pytest.mark.parametrize("nx,ny,nz", [(30, 25, 27), (33, 32, 21)])
def test_projection_after_a_change_of_mask(role, nx, ny, nz):
    pc = {"net": F.FS_PRECOND_LEARNED, "net_mg": F.FS_PRECOND_LEARNED_MG}[role]
    masks = [W.ellipsoid_blob(nx, ny, nz, 1)[0], W.sphere_union(nx, ny, nz, 2, occ_range=(0.05, 0.9))[0],
             W.all_liquid(nx, ny, nz)]
    kw = dict(dx=1.0 / ny, tol_p=1e-6, precond=pc, maxit_p=2000)
    kept = F.Grid(nx, ny, nz, **kw)
    F.fs_net_load(kept.ctx, T.role_weights(role))
    u0 = W.random_mac(nx, ny, nz, 5)
    for types in masks:
        kept.set_mask(types)
        u = kept.pack(u0)
        rc, st = kept.project(u)
        assert rc == F.FS_OK and st["true_relres_p"] <= 1e-6
        fresh = F.Grid(nx, ny, nz, **kw)
        F.fs_net_load(fresh.ctx, T.role_weights(role))
        fresh.set_mask(types)
        v = fresh.pack(u0)
        rc, sf = fresh.project(v)
        # the same operations on the same values
        assert rc == F.FS_OK and sf["iters_p"] == st["iters_p"] and sf["fallbacks"] == st["fallbacks"]
        assert all(torch.equal(a, b) for a, b in zip(u, v))
        ou, _, _ = O.project(O.Grid(types, 1.0 / ny, 1 / 30, 0.01), u0)
        err = sum(float(((a - b) ** 2).sum()) for a, b in zip(kept.unpack(u), ou))
        assert err <= 1e-5 ** 2 * sum(float((b ** 2).sum()) for b in ou)
