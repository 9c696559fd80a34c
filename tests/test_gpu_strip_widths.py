"""The streamed 2-D kernel on widths that are no multiple of its strip: a last
strip with few columns, rows that do not start on 16-byte boundaries, grids
narrower than a strip, unaligned pointers.  Tolerances are those of the whole
strips: 1e-13 / 2e-6 for Q v (Section 2), and for samples the tolerance asked for
with the library's status contract (tests/honesty.py)."""
import numpy as np
import pytest

from honesty import assert_honest
from oracle import lanczos as olz
from oracle import stencil
from paper_1312_1476_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# widths: one column in the last strip, one missing, odd, even but not whole 16 bytes, whole 16 bytes, half a strip
SHAPES = [(512, 129), (260, 255), (301, 383), (264, 250), (256, 260), (1031, 64), (1040, 65)]


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _problem(shape, bc, op, precision, k2):
    from paper_1312_1476_gb300 import gmrf
    return gmrf.Problem(shape, bc, op, kappa2=torch.from_numpy(k2).cuda(), kappa2_const=0.3, precision=precision)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%dx%d" % s)
@pytest.mark.parametrize("bc", ["periodic", "neumann", "dirichlet"])
@pytest.mark.parametrize("op", ["shifted_laplacian", "spde_squared", "spde_plus_diag"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_apply(shape, bc, op, precision):
    dt = np.float64 if precision == "fp64" else np.float32
    n = int(np.prod(shape))
    k2 = inputs.kappa2_uniform_field(shape, seed=4, lo=0.05, hi=1.0)
    Q = stencil.precision_matrix(shape, bc, op, k2.astype(np.float64), 1.0,
                                 **({"kappa2_prior": 0.3} if op == "spde_plus_diag" else {}))
    V = inputs.gaussian_vectors(2, n, seed=5, dtype=dt)
    with _problem(shape, bc, op, precision, k2) as p:
        for shift in (0, 1):  # the second time from and to pointers on no 16-byte boundary
            v = torch.zeros(2 * n + shift, dtype=torch.from_numpy(V).dtype, device="cuda")
            v[shift:] = torch.from_numpy(V.reshape(-1))
            y = torch.zeros_like(v)
            p.apply(0, v[shift:], y[shift:], nvec=2)
            Y = y[shift:].cpu().numpy().reshape(2, n)
            for s in range(2):
                assert _rel(Y[s], Q @ V[s].astype(np.float64)) <= (1e-13 if precision == "fp64" else 2e-6)


@pytest.mark.parametrize("shape,bc,op", [((257, 259), "periodic", "shifted_laplacian"),
                                         ((300, 226), "dirichlet", "shifted_laplacian"),
                                         ((261, 255), "neumann", "spde_squared"),
                                         ((300, 252), "neumann", "shifted_laplacian")])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_samples(shape, bc, op, precision):
    from paper_1312_1476_gb300 import gmrf
    dt = np.float64 if precision == "fp64" else np.float32
    n = int(np.prod(shape))
    k2 = inputs.kappa2_uniform_field(shape, seed=3, lo=0.5 if op == "spde_squared" else 0.05, hi=1.0)
    Q = stencil.precision_matrix(shape, bc, op, k2.astype(np.float64), 1.0)
    Z = inputs.gaussian_vectors(3, n, seed=4, dtype=dt)
    tol = 1e-10 if precision == "fp64" else 1e-6
    with _problem(shape, bc, op, precision, k2) as p:
        x = torch.empty(3 * n, dtype=torch.from_numpy(Z).dtype, device="cuda")
        rc, info = p.sample(x, nsamples=3, tol=tol, m_max=3000, z=torch.from_numpy(Z).cuda(), raise_on_error=False)
        assert rc == gmrf.OK or (precision == "fp32" and rc == gmrf.ERR_NOT_CONVERGED)
        x1 = torch.empty(n, dtype=x.dtype, device="cuda")
        p.sample(x1, nsamples=1, tol=tol, m_max=3000, z=torch.from_numpy(Z[2]).cuda(), raise_on_error=False)
        assert torch.equal(x1, x.reshape(3, n)[2])  # alone as in the batch
        X = x.cpu().numpy().reshape(3, n)
    xe, m, est, st = olz.adaptive_sample(lambda v: Q @ v, Z[0].astype(np.float64), 1e-12, 3000, reorth=True)
    assert st == "ok"
    assert_honest(info[0], _rel(X[0], xe), 1e-9 if precision == "fp64" else 1e-6)
