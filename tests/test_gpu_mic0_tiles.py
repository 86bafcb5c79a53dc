"""MIC(0) substitution where its tiles can go wrong: the smallest grid, one tile, one cell into a
second tile on each axis, and scattered masks with empty tiles, against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2503_00868_gb300 import fluidstep as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_00868_gb300 import build as B
    B.build()
    O.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("nx,ny,nz,liquid", [(2, 2, 2, 1.0), (8, 8, 8, 1.0), (9, 8, 8, 0.9), (8, 9, 17, 0.7), (17, 24, 9, 0.4),
                                             (63, 41, 34, 0.02), (40, 64, 33, 0.8)])
def test_mic0_tiles_match_oracle(nx, ny, nz, liquid):
    rng = np.random.default_rng(7)
    types = np.where(rng.random((nz, ny, nx)) < liquid, 1, 0).astype(np.uint8)
    types.flat[0] = 1
    og = O.Grid(types, 1.0 / ny, 1 / 30, 0.01)
    g = F.Grid(nx, ny, nz, dx=1.0 / ny, precond=F.FS_PRECOND_MIC0)
    g.set_mask(types)
    r = np.where(types == 1, rng.standard_normal(types.shape), 0.0)
    want = O.mic0_apply(og, O.mic0_factor(og), r)
    z = g.empty_cell()
    for _ in range(2):  # the second pair of sweeps starts from counters the first one left
        g.precond_apply(g.pack_cell(r), z)
        # the substitution is a stable recurrence in 32 bits: some hundred roundings of 2^-24 at most
        assert np.linalg.norm(g.unpack_cell(z) - want) <= 1e-5 * max(np.linalg.norm(want), 1e-30)
