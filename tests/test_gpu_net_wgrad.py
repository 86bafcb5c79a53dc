"""The network's weight and bias gradients on the tensor cores against the oracle's
backpropagation, at the edges of the 32 x 8 x 1 tiles the contraction walks: exact
tiles, one cell more and one cell fewer on each axis, several tiles per block."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2503_00868_gb300 import fluidstep as F

from test_gpu_net import rand_params, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(32, 8, 3), (33, 9, 4), (31, 7, 2), (65, 17, 9), (2, 2, 2), (40, 40, 40)])
def test_weight_gradients_at_tile_edges(nx, ny, nz):
    rng = np.random.default_rng(nx * ny * nz)
    types = (rng.random((nz, ny, nx)) < 0.8).astype(np.uint8)
    types[0, 0, 0] = 1
    og = O.Grid(types, 1.0 / ny, 1 / 30, 0.01)
    gg = F.Grid(nx, ny, nz, dx=1.0 / ny)
    gg.set_mask(types)
    flat, Ws, Bs = rand_params(3)
    F.fs_net_load(gg.ctx, flat)
    b, q = (np.where(types == 1, rng.standard_normal(types.shape), 0.0) for _ in range(2))
    F.fs_net_grad(gg.ctx, gg.pack_cell(b), gg.pack_cell(q))
    g = F.fs_net_grad_read(gg.ctx)
    _, gW, gB = O.net_loss_grad(og, Ws, Bs, b, q)
    off = 0
    for w, bias in zip(gW, gB):
        for want in (w.ravel(), np.ravel(bias)):
            # activations and their gradients that fall on the other side of a bf16 rounding differ by
            # 2^-8 of themselves; the sums here are exact to far less
            assert rel(g[off:off + want.size], want) <= 2.0 ** -8
            off += want.size
    assert off == g.size
