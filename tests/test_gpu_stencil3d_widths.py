"""The 3-D kernels that take any width, boundary, precision and pointer alignment
(flat ranges up to 512 wide, tiles beyond): ranges that end inside a row and with
the plane, planes smaller than a range, periodic wraps of two planes.  Tolerances as for the other
stencil kernels: 1e-13 / 2e-6 for Q v (Section 2), for samples the tolerance asked
for with the library's status contract (tests/honesty.py)."""
import numpy as np
import pytest

from honesty import assert_honest
from oracle import lanczos as olz
from oracle import stencil
from paper_1312_1476_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(2, 2, 2), (3, 9, 129), (13, 8, 127), (9, 17, 65), (33, 10, 63), (2, 25, 260), (40, 3, 5), (5, 16, 256),
          (4, 11, 513), (3, 9, 645), (6, 7, 512), (3, 37, 55)]


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%dx%dx%d" % s)
@pytest.mark.parametrize("bc", ["periodic", "neumann", "dirichlet"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_apply(shape, bc, precision):
    from paper_1312_1476_gb300 import gmrf
    dt = np.float64 if precision == "fp64" else np.float32
    n = int(np.prod(shape))
    k2 = inputs.kappa2_uniform_field(shape, seed=4, lo=0.05, hi=1.0)
    V = inputs.gaussian_vectors(2, n, seed=5, dtype=dt)
    for field in (k2, None):  # a field, and a constant
        Q = stencil.precision_matrix(shape, bc, "shifted_laplacian", 0.3 if field is None else k2.astype(np.float64), 1.0)
        with gmrf.Problem(shape, bc, "shifted_laplacian", kappa2=None if field is None else torch.from_numpy(k2).cuda(),
                          kappa2_const=0.3, precision=precision) as p:
            for shift in (0, 1):  # the second time from and to pointers on no 16-byte boundary
                v = torch.zeros(2 * n + shift, dtype=torch.from_numpy(V).dtype, device="cuda")
                v[shift:] = torch.from_numpy(V.reshape(-1))
                y = torch.zeros_like(v)
                p.apply(0, v[shift:], y[shift:], nvec=2)
                Y = y[shift:].cpu().numpy().reshape(2, n)
                for s in range(2):
                    assert _rel(Y[s], Q @ V[s].astype(np.float64)) <= (1e-13 if precision == "fp64" else 2e-6)


@pytest.mark.parametrize("shape,bc", [((11, 13, 37), "dirichlet"), ((9, 20, 130), "periodic"), ((17, 9, 67), "neumann"),
                                      ((4, 9, 517), "dirichlet"), ((4, 8, 530), "periodic")])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_samples(shape, bc, precision):
    from paper_1312_1476_gb300 import gmrf
    dt = np.float64 if precision == "fp64" else np.float32
    n = int(np.prod(shape))
    k2 = inputs.kappa2_uniform_field(shape, seed=3, lo=0.05, hi=1.0)
    Q = stencil.precision_matrix(shape, bc, "shifted_laplacian", k2.astype(np.float64), 1.0)
    Z = inputs.gaussian_vectors(3, n, seed=4, dtype=dt)
    tol = 1e-10 if precision == "fp64" else 1e-6
    with gmrf.Problem(shape, bc, "shifted_laplacian", kappa2=torch.from_numpy(k2).cuda(), precision=precision) as p:
        x = torch.empty(3 * n, dtype=torch.from_numpy(Z).dtype, device="cuda")
        rc, info = p.sample(x, nsamples=3, tol=tol, m_max=1000, z=torch.from_numpy(Z).cuda(), raise_on_error=False)
        assert rc == gmrf.OK or (precision == "fp32" and rc == gmrf.ERR_NOT_CONVERGED)
        x1 = torch.empty(n, dtype=x.dtype, device="cuda")
        p.sample(x1, nsamples=1, tol=tol, m_max=1000, z=torch.from_numpy(Z[2]).cuda(), raise_on_error=False)
        assert torch.equal(x1, x.reshape(3, n)[2])  # alone as in the batch
        if precision == "fp32":  # a bfloat16 basis: the same iteration, element stores
            xb = torch.empty(n, dtype=x.dtype, device="cuda")
            _, ib = p.sample(xb, nsamples=1, tol=tol, m_max=1000, z=torch.from_numpy(Z[2]).cuda(), v_storage="bf16",
                             raise_on_error=False)
            assert ib[0].m_used == info[2].m_used and _rel(xb.cpu().numpy(), x1.cpu().numpy()) <= 1e-2
        X = x.cpu().numpy().reshape(3, n)
    xe, m, est, st = olz.adaptive_sample(lambda v: Q @ v, Z[0].astype(np.float64), 1e-12, 1000, reorth=True)
    assert st == "ok"
    assert_honest(info[0], _rel(X[0], xe), 1e-9 if precision == "fp64" else 1e-6)
