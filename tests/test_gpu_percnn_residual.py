"""The residual that the recurrent solver reports is summed in 64 bits across threads: on
isolated liquid cells with whole velocities of two scales every square, and every sum of
them, is a 53-bit number, so the reported ratio is exact but for its quotient and root."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2503_00868_gb300 import fluidstep as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_residual(seed):
    nx, ny, nz = 65, 65, 65
    rng = np.random.default_rng(seed)
    types = np.zeros((nz, ny, nx), np.uint8)
    types[1::2, 1::2, 1::2] = 1
    side = types[1::2, 1::2, ::2]  # the x neighbours of the liquid
    side[rng.random(side.shape) < 0.3] = 2
    types[1::2, 1::2, ::2] = side
    liq = types == 1
    d = sum(np.roll(np.pad(types != 2, 1), s, a)[1:-1, 1:-1, 1:-1].astype(int) for a in range(3) for s in (1, -1))
    # b = whole numbers below 1024, half of the cells at 2^-8 of them: one velocity, on the lower z face (fluid)
    whole = rng.integers(1, 1024, types.shape)
    shift = np.where(rng.random(types.shape) < 0.5, 8, 0)
    b = np.where(liq, whole * 2.0 ** -shift, 0.0)
    w = np.zeros((nz + 1, ny, nx))
    w[:-1] = b
    g = F.Grid(nx, ny, nz, dx=1.0, pressure_solver=F.FS_SOLVER_PERCNN)
    k = np.zeros(27)
    k[13] = 0.125  # one sub-step: p = b / 8, and the residual is b (8 - d) / 8
    F.fs_percnn_load(g.ctx, k, 1)
    g.set_mask(types)
    rc, st = g.project(g.pack([np.zeros((nz, ny, nx + 1)), np.zeros((nz, ny + 1, nx)), w]))
    assert rc == F.FS_OK
    sq = [int(v) ** 2 << int(16 - 2 * s) for v, s in zip(whole[liq], shift[liq])]
    bb = sum(sq)
    rr = sum(q * (8 - int(n)) ** 2 for q, n in zip(sq, d[liq]))  # 64 times
    assert max(bb, rr).bit_length() <= 53
    want = Fraction(rr, 64 * bb)
    # a quotient and a root, each rounded once: the square is off by at most 2 (2^-53 + 2^-54) of itself
    got = Fraction(float(st["relres_p"])) ** 2
    assert abs(got / want - 1) <= 2 * (Fraction(1, 2 ** 53) + Fraction(1, 2 ** 54)) + Fraction(1, 2 ** 100)
