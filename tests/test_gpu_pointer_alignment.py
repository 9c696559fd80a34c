"""Callers' device arrays that lie at any element of their type, ``buf[1:]`` for instance: the same bits as aligned
arrays, since only the width of the loads and stores differs.  Problems whose kernels move whole vectors otherwise."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _shifted(values, shift):
    """A copy of values at element `shift` of an allocation, which itself is aligned to far more than a vector."""
    buf = torch.full((values.numel() + shift,), float("nan"), dtype=values.dtype, device="cuda")
    view = buf[shift:]
    view.copy_(values)
    assert view.data_ptr() == buf.data_ptr() + shift * values.element_size()
    return view


def _randn(count, dtype, seed):
    return torch.randn(count, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda", dtype=dtype)


def _same_calls(p, n, dtype, shift, tol):
    """Every call of a preconditioned problem that takes the caller's arrays, aligned and shifted."""
    v, empty = _randn(2 * n, dtype, 3), torch.empty(2 * n, dtype=dtype, device="cuda")
    vs = _shifted(v, shift)

    def both(call, *arrays):
        out, out_s = empty.clone().fill_(float("nan")), _shifted(empty, shift).fill_(float("nan"))
        call(*arrays, out)
        call(*[vs if a is v else a for a in arrays], out_s)
        assert torch.isfinite(out).all() and torch.equal(out, out_s)
        # one of the two aligned
        out_s.fill_(float("nan"))
        call(*arrays, out_s)
        assert torch.equal(out, out_s)
        if arrays:
            out2 = torch.empty_like(out)
            call(*[vs if a is v else a for a in arrays], out2)
            assert torch.equal(out, out2)

    for which in (1, 2):
        both(lambda a, y: p.apply(which, a, y, nvec=2), v)
    both(lambda a, y: p.apply_inv_sqrt_noalloc(a, y, nvec=2), v)
    opts = dict(tol=tol, m_max=200, raise_on_error=False)
    both(lambda a, y: p.sample(y, nsamples=2, z=a, **opts), v)
    both(lambda a, y: p.solve(a, y, nrhs=2, **opts), v)
    both(lambda y: p.sample_logdet(y, nsamples=2, nprobes=2, **opts))


@pytest.mark.parametrize("kind,bc", [("mirror", "neumann"), ("circulant", "periodic"), ("mirror", "dirichlet")])
@pytest.mark.parametrize("precision,shift", [("fp32", 1), ("fp32", 2), ("fp64", 1)])
@pytest.mark.parametrize("shape", [(8, 64), (64, 128), (32, 1024)], ids=lambda s: "%dx%d" % s)
def test_squared_operator_on_shifted_arrays(shape, precision, shift, kind, bc):
    from paper_1312_1476_gb300 import gmrf
    f64 = precision == "fp64"
    g = torch.Generator(device="cuda").manual_seed(1)
    k2 = torch.rand(shape, generator=g, device="cuda") + 0.5
    with gmrf.Problem(shape, bc, "spde_squared", kappa2=k2, tau=1.3, precond=kind, precision=precision) as p:
        _same_calls(p, shape[0] * shape[1], torch.float64 if f64 else torch.float32, shift, 1e-9 if f64 else 1e-5)


@pytest.mark.parametrize("kind,bc", [("mirror", "neumann"), ("circulant", "periodic"), ("mirror", "dirichlet")])
@pytest.mark.parametrize("shift", [1, 2])
@pytest.mark.parametrize("shape", [(128, 128), (128, 1024), (256, 2048)], ids=lambda s: "%dx%d" % s)
def test_shifted_laplacian_on_shifted_arrays(shape, shift, kind, bc):
    from paper_1312_1476_gb300 import gmrf
    g = torch.Generator(device="cuda").manual_seed(2)
    k2 = torch.rand(shape, generator=g, device="cuda") + 0.5
    with gmrf.Problem(shape, bc, "shifted_laplacian", kappa2=k2, tau=0.7, precond=kind) as p:
        _same_calls(p, shape[0] * shape[1], torch.float32, shift, 1e-5)


@pytest.mark.parametrize("bc", ["periodic", "neumann", "dirichlet"])
@pytest.mark.parametrize("precision,shift", [("fp32", 1), ("fp32", 2), ("fp64", 1)])
@pytest.mark.parametrize("nx", [516, 518, 1024])
def test_wide_3d_product_on_shifted_arrays(nx, precision, shift, bc):
    from paper_1312_1476_gb300 import gmrf
    shape, n = (5, 9, nx), 45 * nx
    dtype = torch.float64 if precision == "fp64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(4)
    k2 = torch.rand(shape, generator=g, device="cuda") + 0.5
    v = _randn(2 * n, dtype, 6)
    with gmrf.Problem(shape, bc, "shifted_laplacian", kappa2=k2, precision=precision) as p:
        want = torch.empty_like(v)
        p.apply(0, v, want, nvec=2)
        for a, y in ((_shifted(v, shift), torch.empty_like(v)), (v, _shifted(v, shift)),
                     (_shifted(v, shift), _shifted(v, shift))):
            p.apply(0, a, y.fill_(float("nan")), nvec=2)
            # one cell a thread instead of two or four: up to eleven roundings of terms of at most 8 max |v|
            assert (y - want).abs().max() <= 12 * 13.5 * torch.finfo(dtype).eps * v.abs().max()


def test_server_writes_shifted_arrays():
    from paper_1312_1476_gb300 import gmrf
    shape, n = (64, 64), 4096
    with gmrf.Problem(shape, "neumann", "spde_squared", kappa2_const=0.3, precond="mirror") as p:
        want = torch.empty(3 * n, device="cuda")
        p.sample(want, nsamples=3, seed=5, m_max=200)
        got = _shifted(torch.zeros_like(want), 1)
        with gmrf.Server(p, nslots=4, m_max=200) as sv:
            req = sv.submit_sample(got, 3, 5)
            for _ in range(1000):
                if sv.step() == 0:
                    break
            assert sv.poll(req) is not None
    assert torch.equal(got, want)
