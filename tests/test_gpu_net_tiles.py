"""Network inference at the edges of its 32 x 8 x 4 tiles against the oracle: exact
tiles, one cell more and one fewer per axis, more tiles than blocks, and an output
that is zero off the liquid; repeated, since a second pass finds other buffers."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2503_00868_gb300 import fluidstep as F

from test_gpu_net import rand_params, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,fill", [(32, 8, 4, 0.8), (33, 9, 5, 0.8), (31, 7, 3, 0.8), (65, 17, 9, 0.02),
                                           (2, 2, 2, 1.0), (96, 64, 30, 0.6)])
def test_inference_at_tile_edges(nx, ny, nz, fill):
    rng = np.random.default_rng(nx + ny + nz)
    types = (rng.random((nz, ny, nx)) < fill).astype(np.uint8)
    types[-1, -1, -1] = 1
    og = O.Grid(types, 1.0 / ny, 1 / 30, 0.01)
    gg = F.Grid(nx, ny, nz, dx=1.0 / ny)
    gg.set_mask(types)
    flat, Ws, Bs = rand_params(4)
    F.fs_net_load(gg.ctx, flat)
    z = gg.empty_cell()
    for _ in range(2):
        r = np.where(types == 1, rng.standard_normal(types.shape), 0.0)
        F.fs_net_forward(gg.ctx, gg.pack_cell(r), z)
        got = gg.unpack_cell(z)
        # an activation on the other side of a bf16 rounding differs by 2^-8 of itself
        assert rel(got, O.net_forward(og, Ws, Bs, r)) <= 2.0 ** -8
        assert np.all(got[types != 1] == 0.0)
