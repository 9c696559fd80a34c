"""Small 2-D grids, whose Lanczos steps run in one launch of a thread-block cluster per vector while
there are few vectors: the same bits as one launch per step, which serves many vectors and is held
to the oracle elsewhere.  The sizes lie at the edges of the tiles (32 columns; 8 rows in FP64, 16 in
FP32), of the clusters (1, 2, 3, 16, 17, 64 and 65 tiles) and of the grid's own boundaries."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(2, 5), (8, 32), (9, 33), (7, 65), (24, 24), (64, 64), (16, 257), (136, 32), (17, 250), (67, 100), (128, 128),
         (130, 121), (255, 63), (520, 32), (1024, 32)]


def _problem(shape, bc, precision, field):
    from paper_1312_1476_gb300 import gmrf
    g = torch.Generator(device="cuda").manual_seed(7)
    k2 = (torch.rand(shape, generator=g, device="cuda") + 0.2) if field else None
    return gmrf.Problem(shape, bc=bc, op="shifted_laplacian", kappa2=k2, kappa2_const=0.2, precision=precision)


@pytest.mark.parametrize("store", ["fp32", "bf16", "fp64"])
@pytest.mark.parametrize("bc,field", [("periodic", False), ("periodic", True), ("neumann", True), ("dirichlet", False)])
@pytest.mark.parametrize("shape", SIZES)
def test_few_vectors_as_in_a_batch(shape, bc, field, store):
    n = shape[0] * shape[1]
    dt, precision = (torch.float64, "fp64") if store == "fp64" else (torch.float32, "fp32")
    tol = 1e-9 if store == "fp64" else 1e-5
    tiles = -(-shape[1] // 32) * -(-shape[0] // (8 if store == "fp64" else 16))
    many = 5 * 152 // tiles + 1
    g = torch.Generator(device="cuda").manual_seed(n)
    z = torch.randn(many, n, generator=g, device="cuda", dtype=dt)
    opts = dict(tol=tol, m_max=120, raise_on_error=False)
    kept = dict(v_storage="bf16") if store == "bf16" else {}
    batch, few = torch.empty_like(z), torch.empty_like(z[:2])
    with _problem(shape, bc, precision, field) as p:
        _, info = p.sample(batch, nsamples=many, z=z, **opts, **kept)
        want = [(i.m_used, i.status) for i in info[:2]]
        for host_loop, every in ((False, 16), (True, 16), (True, 1)):
            p.set_tuning(host_loop=host_loop)
            few.fill_(float("nan"))
            _, info = p.sample(few, nsamples=2, z=z[:2], check_every=every, **opts, **kept)
            assert [(i.m_used, i.status) for i in info] == want
            assert torch.equal(few, batch[:2])
        p.set_tuning()
        p.solve(z, batch, nrhs=many, **opts)
        p.solve(z[:2], few, nrhs=2, **opts)
        assert torch.equal(few, batch[:2])
        q = p.logdet(nprobes=many, probes=z, **opts)[2]
        assert (p.logdet(nprobes=2, probes=z[:2], **opts)[2] == q[:2]).all()
