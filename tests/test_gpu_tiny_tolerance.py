"""Tolerances whose square underflows: the stopping rule compares squares, and must not take two that are 0 for
convergence.  kappa^2 = 8 makes the condition of the 5-point operator 2, so that the recurrence's residual, which goes on
falling below the rounding level, passes 1e-162, where its square is 0, and then 1e-200 within a few hundred steps; what a
vector stops with is the residual there, which is not 0."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-200


# one vector: all steps in one launch; 900: a launch a step
@pytest.mark.parametrize("shape,nvec", [((64, 64), 1), ((24, 24), 900), ((256, 256), 1), ((12, 20, 16), 2)])
def test_not_before_the_residual_is_there(shape, nvec):
    from paper_1312_1476_gb300 import gmrf
    n = math.prod(shape)
    b = torch.randn(nvec, n, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda", dtype=torch.float64)
    x = torch.empty_like(b)
    with gmrf.Problem(shape, "periodic", "shifted_laplacian", kappa2_const=8.0, precision="fp64") as p:
        rc, info = p.solve(b, x, nrhs=nvec, tol=TOL, m_max=500)
        probes = p.logdet(nprobes=min(nvec, 4), probes=b.sign(), tol=TOL, m_max=500)[3]
    assert rc == gmrf.OK
    for i in list(info) + list(probes):
        assert i.status == gmrf.OK and 0 < i.err_est <= TOL
