"""P2G's ordering memory has room for a count that rises from call to call: up to an
eighth more particles take no new memory, and what is kept is given back with the
context."""
import pytest
import torch

from paper_2503_00868_gb300 import fluidstep as F

pytestmark = pytest.mark.gpu


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_rising_count():
    n, k = 32, 2_000_000  # 128 MB of records
    most = k + k // 8
    x = 0.1 + 0.8 * torch.rand(most, 3, device="cuda")  # every node that a particle reaches is in the grid
    v, C, m = torch.randn(most, 3, device="cuda"), torch.zeros(most, 9, device="cuda"), torch.ones(most, device="cuda")
    warm = F.Grid(n, n, n, dx=1.0 / n)  # kernels loaded, torch's own pool settled
    u, mass = warm.zeros(), warm.zeros()
    F.fs_p2g(warm.ctx, x[:1000], v[:1000], C[:1000], m[:1000], u, mass)
    F.fs_p2g(warm.ctx, x, v, C, m, u, mass)
    warm.close()
    float(mass.u.sum())
    at_start = free()
    g = F.Grid(n, n, n, dx=1.0 / n)
    F.fs_p2g(g.ctx, x[:k], v[:k], C[:k], m[:k], u, mass)
    kept = free()
    assert at_start - kept >= 64 * k
    for c in (k + 1, k + k // 16, most):
        F.fs_p2g(g.ctx, x[:c], v[:c], C[:c], m[:c], u, mass)
        assert free() == kept
        assert abs(float(mass.u.sum()) / c - 1) < 1e-3
    F.fs_p2g(g.ctx, x[:70000], v[:70000], C[:70000], m[:70000], u, mass)
    assert free() == kept
    g.close()
    assert free() >= at_start
