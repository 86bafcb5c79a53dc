"""A solve that could not run is the call's error: a projection, a step or a reverse step
does not return success, or a soft status, with a pressure that was not solved for."""
import pytest

from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "no network": (dict(precond=F.FS_PRECOND_LEARNED), F.FS_ESTATE),
    "no network, V-cycle": (dict(precond=F.FS_PRECOND_LEARNED_MG), F.FS_ESTATE),
    "no kernel": (dict(pressure_solver=F.FS_SOLVER_PERCNN), F.FS_ESTATE),
    "wait ran out": (dict(precond=F.FS_PRECOND_MIC0, spin_limit=1), F.FS_ETIMEOUT),
}


@pytest.mark.parametrize("call", ["project", "step", "adjoint"])
@pytest.mark.parametrize("case", sorted(CASES))
def test_status(case, call):
    kw, want = CASES[case]
    n = 48
    g = F.Grid(n, n, n, dx=1.0 / n, nu=0.01, maxit_p=2000, **kw)
    g.set_mask(W.ellipsoid_blob(n, n, n, 0)[0])
    u = g.pack(W.random_mac(n, n, n, 3))
    with pytest.raises(F.FluidStepError) as e:
        if call == "project":
            g.project(u)
        elif call == "step":
            g.step(u, g.zeros())
        else:
            g.adjoint_step(u, g.pack(W.random_mac(n, n, n, 4)), g.zeros())
    assert e.value.status == want
    # the context stays usable
    g.set_params(precond=F.FS_PRECOND_MG, pressure_solver=F.FS_SOLVER_PCG, spin_limit=1 << 22)
    rc, st = g.project(u)
    assert rc == F.FS_OK and st["true_relres_p"] <= 2e-6
