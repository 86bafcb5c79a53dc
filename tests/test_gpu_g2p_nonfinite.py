"""G2P of particles without a finite position: they reach no node, so they take no
velocity and no gradient, keep their deformation and are clamped when they advance;
the particles beside them in the warp are those of a call without them."""
import numpy as np
import pytest
import torch

from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 3e38])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_g2p(bad, axis):
    nx, ny, nz, n, dx = 12, 9, 10, 75, 0.25
    rng = np.random.default_rng(5)
    x = rng.uniform(0.2, 2.0, (n, 3)).astype(np.float32)
    ill = np.array([0, 17, 31, 32, 74])
    x[ill, axis] = bad
    g = F.Grid(nx, ny, nz, dx=dx)
    u = g.pack(W.random_mac(nx, ny, nz, 6))
    dev = lambda a: torch.tensor(np.asarray(a, np.float32), device="cuda")  # noqa: E731
    F0 = (np.eye(3) + 0.1 * rng.standard_normal((n, 3, 3))).reshape(n, 9).astype(np.float32)
    A0 = rng.standard_normal((n, 9)).astype(np.float32)

    def run(xs, keep):
        xt, v, C = dev(xs), torch.full((len(xs), 3), 7.0, device="cuda"), torch.full((len(xs), 9), 7.0, device="cuda")
        Ft, A = dev(F0[keep]), torch.full((len(xs), 9), 7.0, device="cuda")
        F.fs_g2p(g.ctx, xt, v, C, u, F=Ft, A0=dev(A0[keep]), A_out=A, dt=0.02, advance=True, lo=0.1, hi=2.1)
        return [t.cpu().numpy() for t in (xt, v, C, Ft, A)]

    xt, v, C, Ft, A = run(x, np.arange(n))
    assert not v[ill].any() and not C[ill].any()
    assert np.array_equal(Ft[ill], F0[ill])
    f3 = F0[ill].reshape(-1, 3, 3).astype(np.float64)
    want = f3 @ A0[ill].reshape(-1, 3, 3) @ np.transpose(f3, (0, 2, 1))
    assert np.abs(A[ill].reshape(-1, 3, 3) - want).max() <= 16 * 2.0 ** -24 * np.abs(f3).max() ** 2 * np.abs(A0).max() * 9
    at = np.where(np.isnan(bad), 0.1, np.clip(bad, 0.1, 2.1)).astype(np.float32)
    assert (xt[ill, axis] == at).all()
    well = np.setdiff1d(np.arange(n), ill)
    for a, b in zip((xt, v, C, Ft, A), run(x[well], well)):
        assert np.array_equal(a[well], b)
