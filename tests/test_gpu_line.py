"""B_bar^{-1} by a transform along x and a recurrence along y, at the edges of
its range, against the oracle's spectral apply (Section 5.1, Theorem 2).

Tolerances (relative 2-norm, u the unit roundoff): the two transforms along x
contribute at most about 4 u per radix-2 level and direction, the recurrences a
fixed number of roundings per value (two per sweep, log2 of the chunks for the
carries): (8 log2 nx + 4 log2 ny + 32) u.  M^{-1/2} v is compared for smooth and
for steep columns: kappa_bar^2 from 1e-4 (rho close to 1, the ends matter) to 4.
"""
import numpy as np
import pytest

from oracle import lanczos as olz
from oracle import exact, precond, stencil

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu



def _inverse(shape, bc, kb, v):
    """B_bar^{-1} v from the closed-form spectrum, its eigenvalues as 4 sin^2: 2 - 2 cos cancels for the smooth modes
    (an absolute error of an ulp of 2, which at kappa_bar^2 = 1e-4 is 3e-14 of the result), and so does sin(pi - x)."""
    lam = kb
    for d, s in enumerate(shape):
        k = np.arange(s)
        th = np.minimum(k, s - k) * (np.pi / s) if bc == "periodic" else k * (np.pi / (2 * s))
        lam = lam + (4 * np.sin(th) ** 2).reshape([-1 if e == d else 1 for e in range(2)])
    return exact.spectral_apply(shape, bc, 1.0 / lam, v)


SHAPES = [(8, 64), (16, 64), (32, 128), (64, 256), (128, 64), (8, 4096), (256, 512), (512, 128), (1024, 64),
          (2048, 64), (4096, 64), (128, 1024), (64, 2048)]


@pytest.mark.parametrize("kind,bc", [("circulant", "periodic"), ("mirror", "neumann")])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%dx%d" % s)
def test_inverse_by_lines(shape, kind, bc, precision):
    from paper_1312_1476_gb300 import gmrf
    f64 = precision == "fp64"
    u = np.finfo(np.float64 if f64 else np.float32).eps / 2
    tol = (8 * np.log2(shape[1]) + 4 * np.log2(shape[0]) + 32) * u
    n = shape[0] * shape[1]
    V = np.random.default_rng(5).standard_normal((3, n)).astype(np.float64 if f64 else np.float32)
    for kb in (1e-4, 0.05, 4.0):
        with gmrf.Problem(shape, bc, "spde_squared", kappa2_const=kb, precond=kind, precision=precision) as p:
            y = torch.empty((3, n), dtype=torch.float64 if f64 else torch.float32, device="cuda")
            p.apply(2, torch.from_numpy(V).cuda(), y, nvec=3)
        for s in range(3):
            ref = _inverse(shape, bc, kb, V[s].astype(np.float64))
            err = np.linalg.norm(y[s].cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err <= tol, (kb, s, err, tol)


@pytest.mark.parametrize("kind,bc", [("periodic", "neumann"), ("periodic", "dirichlet"), ("neumann", "dirichlet"),
                                     ("neumann", "periodic")])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", [(8, 64), (32, 256), (16, 2048)], ids=lambda s: "%dx%d" % s)
def test_operator_with_boundary_terms(shape, kind, bc, precision):
    """A v where the boundaries of M and Q differ (partner rows of other blocks, lines in and across warps).
    Two solves, each within the bound above, act on vectors of the size of w = B_bar^{-1} v; R multiplies by at most
    8 + max kappa^2 and ||B_bar^{-1}|| <= 1 / kappa_bar^2, once per factor of A = C^T C."""
    from paper_1312_1476_gb300 import gmrf
    f64 = precision == "fp64"
    u = np.finfo(np.float64 if f64 else np.float32).eps / 2
    n = shape[0] * shape[1]
    rng = np.random.default_rng(7)
    k2 = rng.uniform(0.5, 1.5, shape).astype(np.float32)
    kb = precond.kappa2_bar(k2)
    A = olz.preconditioned_operator(stencil.precision_matrix(shape, bc, "spde_squared", k2.astype(np.float64), tau=1.0),
                                    shape, kind, "spde_squared", kb, 1.0)
    v = rng.standard_normal(n).astype(np.float64 if f64 else np.float32)
    with gmrf.Problem(shape, bc, "spde_squared", kappa2=torch.from_numpy(k2).cuda(),
                      precond="circulant" if kind == "periodic" else "mirror", kappa2_precond=kb,
                      precision=precision) as p:
        y = torch.empty(n, dtype=torch.float64 if f64 else torch.float32, device="cuda")
        p.apply(1, torch.from_numpy(v).cuda(), y)
    ref = A(v.astype(np.float64))
    gain = (1 + 9.5 / kb) ** 2
    tol = gain * (8 * np.log2(shape[1]) + 4 * np.log2(shape[0]) + 32) * u
    assert np.linalg.norm(y.cpu().numpy() - ref) / np.linalg.norm(v) <= tol
