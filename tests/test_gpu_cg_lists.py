"""The CG kernels over lists of active quads with the Jacobi and MIC(0) preconditioners:
lone quads, broken rows and a ragged full box, against the oracle's step."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_00868_gb300 import build as B
    B.build()
    O.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("precond", [F.FS_PRECOND_JACOBI, F.FS_PRECOND_MIC0])
@pytest.mark.parametrize("nx,ny,nz,liquid", [(2, 2, 2, 0.5), (37, 21, 18, 0.04), (64, 9, 33, 0.5), (31, 30, 29, 1.0)])
def test_step_over_lists_matches_oracle(nx, ny, nz, liquid, precond):
    types = np.where(np.random.default_rng(2).random((nz, ny, nx)) < liquid, 1, 0).astype(np.uint8)
    types.flat[0] = 1
    if liquid == 1.0:
        types[:, -1, :] = 0  # an open surface
    u0 = W.blurred_noise_mac(nx, ny, nz, 4)
    og = O.Grid(types, 1.0 / ny, 1 / 30, 0.01)
    g = F.Grid(nx, ny, nz, dx=1.0 / ny, dt=1 / 30, nu=0.01, tol_p=1e-7, tol_v=1e-7, precond=precond)
    g.set_mask(types)
    want, _ = O.step(og, u0)
    out = g.zeros()
    rc, _ = g.step(g.pack(u0), out)
    assert rc == F.FS_OK
    got = g.unpack(out)
    num = sum(float(((a - b) ** 2).sum()) for a, b in zip(got, want)) ** 0.5
    den = sum(float((b ** 2).sum()) for b in want) ** 0.5
    # the bound of the other comparisons of a step with the oracle at this tolerance
    assert num <= 1e-5 * den
