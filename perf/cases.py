"""The calls whose speed counts: what a program that uses this library has it do.

Every case goes through the public binding (``paper_1312_1476_gb300.gmrf``).  The kinds:

``inv_sqrt``   y = M^{-1/2} v of the constant-coefficient preconditioner, called by itself
``apply``      y = Q v, the matrix-vector product of a caller's own solver
``sample``     x = Q^{-1/2} z of a lattice, with or without the preconditioner
``solve``      x = Q^{-1} b, preconditioned
``logdet``     the Hutchinson / Lanczos quadratures of log det Q
``block``      samples and log-det probes in one block of vectors
``proposal``   the two linear-algebra calls of one sMMALA proposal: a solve and a sample
``sparse``     samples of a general sparse Q with an incomplete-Cholesky factor
``serve``      the slot server on a handful of requests

Sizes are those of the benchmark configurations and of the tests.  ``z``, probes and right-hand
sides are handed in on the device, as a program does that has its own noise; the server draws its own.
"""
import math

import numpy as np
import torch

from paper_1312_1476_gb300 import gmrf


def listed():
    return [
        # a caller's own iteration applies the prior's factor to one small field: launches and latency only
        dict(name="inv_sqrt_128", kind="inv_sqrt", ny=128, nx=128, nvec=1, precision="fp32", precond="mirror"),
        # the exact-arithmetic check problem, one draw at 1e-10: 4096 cells in FP64, about a hundred dependent steps
        dict(name="sample_64_f64", kind="sample", nz=0, ny=64, nx=64, bc="periodic", op="shifted_laplacian",
             field="const", precond="none", precision="fp64", nvec=1, tol=1e-10, m_max=300),
        # the same lattice when a study wants many draws of it
        dict(name="sample_64_f64_x256", kind="sample", nz=0, ny=64, nx=64, bc="periodic", op="shifted_laplacian",
             field="const", precond="none", precision="fp64", nvec=256, tol=1e-10, m_max=300),
        # the headline: one draw of a million-cell SPDE field
        dict(name="sample_1024", kind="sample", nz=0, ny=1024, nx=1024, bc="neumann", op="spde_squared",
             field="smooth", precond="mirror", precision="fp32", nvec=1, tol=1e-6, m_max=200),
        # a Monte Carlo study: 256 draws and 64 log-det probes of one field in one call
        dict(name="block_512", kind="block", ny=512, nx=512, nvec=256, nprobes=64, tol=1e-6, m_max=100),
        # one sMMALA proposal of the log-Gaussian Cox process, in FP64 to 1e-8
        dict(name="proposal_512_f64", kind="proposal", ny=512, nx=512, precision="fp64", tol=1e-8, m_max=64),
        # the 13-point product on a block of vectors, for a solver that is the caller's own
        dict(name="apply_q_1024_x16", kind="apply", nz=0, ny=1024, nx=1024, bc="neumann", op="spde_squared",
             field="smooth", precision="fp32", nvec=16),
        # an observation window of odd size, no preconditioner: log det of the 5-point operator
        dict(name="logdet_701x999", kind="logdet", nz=0, ny=701, nx=999, bc="periodic", op="shifted_laplacian",
             field="const", precond="none", precision="fp32", nvec=16, tol=1e-6, m_max=200),
        # a small three-dimensional field of odd size
        dict(name="sample_3d_odd", kind="sample", nz=61, ny=75, nx=90, bc="dirichlet", op="shifted_laplacian",
             field="uniform", precond="none", precision="fp32", nvec=4, tol=1e-6, m_max=100),
        # the large three-dimensional field: eight draws, the basis alone is tens of gigabytes
        dict(name="sample_3d_256_x8", kind="sample", nz=256, ny=256, nx=256, bc="dirichlet", op="shifted_laplacian",
             field="uniform", precond="none", precision="fp32", nvec=8, tol=1e-6, m_max=48),
        # the general sparse matrix of the paper's Figure 3 with a thresholded factor, many draws
        dict(name="figure3_ict_x256", kind="sparse", side=30, droptol=1e-3, shift=1e-3, precision="fp64", nvec=256,
             tol=1e-8, m_max=128),
        # requests of several sizes served from one table of slots
        dict(name="serve_256", kind="serve", ny=256, nx=256, slots=24, counts="8,1,20,5", probes=16, tol=1e-6,
             m_max=128),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["inv_sqrt", "apply", "sample_small", "sample_2d", "sample_3d", "sample_pre", "sample_pre",
                       "solve", "logdet", "logdet_pre", "block", "proposal", "sparse", "serve"])
    if kind == "inv_sqrt":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        return dict(kind="inv_sqrt", ny=2 ** rng.randint(5, 11), nx=2 ** rng.randint(5, 11), nvec=_log_int(rng, 1, 16),
                    precision=prec, precond=rng.choice(["mirror", "circulant"]))
    if kind == "apply":
        if rng.random() < 0.3:
            return dict(kind="apply", nz=rng.randint(17, 160), ny=rng.randint(17, 160), nx=rng.randint(17, 160),
                        bc=rng.choice(["dirichlet", "neumann", "periodic"]), op="shifted_laplacian", field="uniform",
                        precision="fp32", nvec=_log_int(rng, 1, 16))
        return dict(kind="apply", nz=0, ny=_log_int(rng, 64, 1500), nx=rng.choice([_log_int(rng, 64, 1500), 512, 1024]),
                    bc=rng.choice(["dirichlet", "neumann", "periodic"]), op=rng.choice(["shifted_laplacian", "spde_squared"]),
                    field="smooth", precision=rng.choice(["fp32", "fp32", "fp64"]), nvec=_log_int(rng, 1, 16))
    if kind == "sample_small":
        return dict(kind="sample", nz=0, ny=rng.randint(24, 130), nx=rng.randint(24, 130),
                    bc=rng.choice(["periodic", "neumann", "dirichlet"]), op="shifted_laplacian", field="const",
                    precond="none", precision="fp64", nvec=_log_int(rng, 1, 128), tol=rng.choice([1e-8, 1e-10]),
                    m_max=300)
    if kind == "sample_2d":
        return dict(kind="sample", nz=0, ny=_log_int(rng, 150, 1200), nx=_log_int(rng, 150, 1200),
                    bc=rng.choice(["periodic", "neumann", "dirichlet"]), op="shifted_laplacian", field="smooth",
                    precond="none", precision="fp32", nvec=_log_int(rng, 1, 8), tol=1e-6, m_max=250)
    if kind == "sample_3d":
        s = [_log_int(rng, 32, 144) for _ in range(3)]
        return dict(kind="sample", nz=s[0], ny=s[1], nx=s[2], bc=rng.choice(["dirichlet", "neumann", "periodic"]),
                    op="shifted_laplacian", field="uniform", precond="none", precision="fp32",
                    nvec=_log_int(rng, 1, 24), tol=1e-6, m_max=100)
    if kind == "sample_pre":
        ny, nx = 2 ** rng.randint(7, 11), 2 ** rng.randint(7, 10)
        return dict(kind="sample", nz=0, ny=ny, nx=nx, bc="neumann", op="spde_squared", field="smooth",
                    precond="mirror", precision="fp32", nvec=_log_int(rng, 1, max(1, min(64, 2 ** 24 // (ny * nx)))),
                    tol=1e-6, m_max=200)
    if kind == "solve":
        ny, nx = 2 ** rng.randint(7, 10), 2 ** rng.randint(7, 11)
        return dict(kind="solve", ny=ny, nx=nx, nvec=_log_int(rng, 1, max(1, min(32, 2 ** 23 // (ny * nx)))),
                    precision="fp32", tol=1e-6, m_max=250)
    if kind == "logdet":
        return dict(kind="logdet", nz=0, ny=_log_int(rng, 200, 1024), nx=_log_int(rng, 200, 1024),
                    bc=rng.choice(["periodic", "dirichlet"]), op="shifted_laplacian", field="const", precond="none",
                    precision="fp32", nvec=rng.randint(4, 24), tol=1e-6, m_max=200)
    if kind == "logdet_pre":
        n = 2 ** rng.randint(7, 9)
        return dict(kind="logdet", nz=0, ny=n, nx=n, bc="neumann", op="spde_squared", field="smooth",
                    precond="mirror", precision="fp32", nvec=rng.randint(4, 64), tol=1e-6, m_max=200)
    if kind == "block":
        return dict(kind="block", ny=2 ** rng.randint(7, 9), nx=2 ** rng.randint(7, 9), nvec=rng.randint(2, 64),
                    nprobes=rng.randint(2, 64), tol=1e-6, m_max=100)
    if kind == "proposal":
        n = 2 ** rng.randint(6, 10)
        prec = rng.choice(["fp32", "fp64", "fp64"])
        return dict(kind="proposal", ny=n, nx=n, precision=prec, tol=1e-6 if prec == "fp32" else rng.choice([1e-6, 1e-8]),
                    m_max=64)
    if kind == "sparse":
        return dict(kind="sparse", side=rng.randint(16, 40), droptol=10.0 ** rng.uniform(-5, -2),
                    shift=10.0 ** rng.uniform(-3, -2), precision="fp64", nvec=_log_int(rng, 1, 256), tol=1e-8,
                    m_max=200)
    n = 2 ** rng.randint(7, 9)
    return dict(kind="serve", ny=n, nx=n, slots=rng.randint(8, 32),
                counts=",".join(str(_log_int(rng, 1, 24)) for _ in range(rng.randint(2, 5))),
                probes=rng.randint(4, 24), tol=1e-6, m_max=128)


# ------------------------------------------------------------------ inputs
MEAN_K2, CONST_K2 = 0.05, 0.1


def _gen(seed, part):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 16 + part)
    return g


def _randn(shape, seed, part, dtype):
    return torch.randn(shape, generator=_gen(seed, part), device="cuda", dtype=dtype)


def _shape(c):
    return (c["nz"], c["ny"], c["nx"]) if c.get("nz") else (c["ny"], c["nx"])


def _smooth(shape, seed, mean, sd, ell):
    """exp of a smooth Gaussian field: white noise filtered with a squared-exponential density, standardised."""
    big = tuple(2 * s for s in shape)
    f2 = sum(f * f for f in torch.meshgrid(*[torch.fft.fftfreq(s, device="cuda", dtype=torch.float64) for s in big],
                                           indexing="ij"))
    f = torch.fft.ifftn(torch.fft.fftn(_randn(big, seed, 1, torch.float64)) * torch.exp(-math.pi ** 2 * ell ** 2 * f2))
    f = f.real[tuple(slice(0, s) for s in shape)]
    return torch.exp(math.log(mean) + sd * (f - f.mean()) / f.std()).float().contiguous()


def _field(c, seed):
    """kappa^2 of the lattice as the configurations draw it, or None for the constant."""
    kind, shape = c.get("field", "smooth"), _shape(c)
    if kind == "const":
        return None
    if kind == "uniform":
        return torch.rand(shape, generator=_gen(seed, 1), device="cuda") * 0.99 + 0.01
    return _smooth(shape, seed, MEAN_K2, 0.5, max(4.0, min(64.0, min(shape) / 16.0)))


def _noise(c, seed, nvec):
    n = int(np.prod(_shape(c)))
    return _randn((nvec, n), seed, 2, torch.float64 if c.get("precision", "fp32") == "fp64" else torch.float32)


def _probes(c, seed, nprobes):
    n = int(np.prod(_shape(c)))
    return torch.randint(0, 2, (nprobes, n), generator=_gen(seed, 3), device="cuda").float().mul_(2).sub_(1)


def _lgcp(c, seed):
    """The proposal's precision on the unit torus, and its gradient: prior (kappa^2 + L / h^2)^2, Poisson counts."""
    N = c["ny"]
    h = 1.0 / N
    lam = _smooth((N, N), seed, 2000.0, 1.0, max(0.1 * N, 1.0)).double()
    mean = h * h * lam
    grad = torch.poisson(mean, generator=_gen(seed, 4)) - mean
    return dict(kc2=100.0 * h * h, tau=1.0 / (h * h), d=(h ** 4 * lam).float().contiguous(), grad=grad.reshape(-1))


_FACTORS = {}


def _figure3(side, droptol, shift):
    """(31^2 G)^2 of a side x side lattice, dense, and a threshold incomplete-Cholesky factor of it: the caller's own matrices."""
    key = (side, droptol, shift)
    if key in _FACTORS:
        return _FACTORS[key]
    t = 2 * np.eye(side) - np.eye(side, k=1) - np.eye(side, k=-1)
    G = 961.0 * (np.kron(np.eye(side), t) + np.kron(t, np.eye(side)))
    Q = G @ G
    n = side * side
    while True:
        A = Q + shift * np.diag(np.diag(Q))
        F = np.zeros((n, n))
        for j in range(n):
            lo = max(0, j - 8 * side)  # no entry of the factor lies further from the diagonal than the matrix's band
            w = A[j:, j] - F[j:, lo:j] @ F[j, lo:j]
            if not w[0] > 0:
                break
            w[1:][np.abs(w[1:]) < droptol * np.abs(A[j:, j]).sum()] = 0.0
            F[j:, j] = w / math.sqrt(w[0])
        else:
            break
        shift *= 4.0
    _FACTORS.clear()
    _FACTORS[key] = (Q, F)
    return _FACTORS[key]


def _csr(M):
    r, k = np.nonzero(M)
    return np.concatenate([[0], np.cumsum(np.bincount(r, minlength=len(M)))]).astype(np.int64), k.astype(np.int32), M[r, k]


def _spde(c, k2):
    return gmrf.Problem((c["ny"], c["nx"]), bc="neumann", op="spde_squared", kappa2=k2, precond="mirror",
                        precision=c.get("precision", "fp32"))


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c}
    prec = c.get("precision", "fp32")
    if kind == "inv_sqrt":
        s["p"] = gmrf.Problem((c["ny"], c["nx"]), bc="neumann" if c["precond"] == "mirror" else "periodic",
                              op="spde_squared", kappa2_const=MEAN_K2, precond=c["precond"], precision=prec)
        s["v"] = _noise(c, seed, c["nvec"])
        s["x"] = torch.empty_like(s["v"])
    elif kind in ("apply", "sample", "logdet"):
        k2 = _field(c, seed)
        s["p"] = gmrf.Problem(_shape(c), bc=c["bc"], op=c["op"], kappa2=k2, kappa2_const=CONST_K2,
                              precond=c.get("precond", "none"), precision=prec)
        if kind == "logdet":
            s["v"] = _probes(c, seed, c["nvec"])
        else:
            s["v"] = _noise(c, seed, c["nvec"])
            s["x"] = torch.empty_like(s["v"])
    elif kind == "solve":
        s["p"] = _spde(c, _field(c, seed))
        s["v"] = _noise(c, seed, c["nvec"])
        s["x"] = torch.empty_like(s["v"])
    elif kind == "block":
        s["p"] = _spde(c, _field(c, seed))
        s["v"] = _noise(c, seed, c["nvec"])
        s["x"] = torch.empty_like(s["v"])
        s["probes"] = _probes(c, seed, c["nprobes"])
    elif kind == "proposal":
        m = _lgcp(c, seed)
        s["p"] = gmrf.Problem((c["ny"], c["nx"]), bc="periodic", op="spde_plus_diag", kappa2=m["d"],
                              kappa2_const=m["kc2"], tau=m["tau"], precond="circulant", precision=prec)
        s["v"] = _noise(c, seed, 1)
        s["b"] = m["grad"].to(s["v"].dtype)
        s["mean"], s["x"] = torch.empty_like(s["b"]), torch.empty_like(s["v"])
    elif kind == "sparse":
        Q, F = _figure3(c["side"], c["droptol"], c["shift"])
        s["p"] = gmrf.SparseProblem(_csr(Q), _csr(F), precision=prec)
        s["v"] = _randn((c["nvec"], c["side"] ** 2), seed, 2, torch.float64)
        s["x"] = torch.empty_like(s["v"])
    elif kind == "serve":
        s["p"] = _spde(c, _field(c, seed))
        s["server"] = gmrf.Server(s["p"], c["slots"], m_max=c["m_max"], tol=c["tol"])
        s["out"] = [torch.empty((int(k), s["p"].n), device="cuda") for k in c["counts"].split(",")]
        s["seed"] = int(seed)
    else:
        raise ValueError(kind)
    return s


def run(state):
    s, c = state, state["case"]
    kind, p = c["kind"], s["p"]
    if kind == "inv_sqrt":
        p.apply(2, s["v"], s["x"], nvec=c["nvec"])
        return s["x"]
    if kind == "apply":
        p.apply(0, s["v"], s["x"], nvec=c["nvec"])
        return s["x"]
    if kind == "sample":
        p.sample(s["x"], nsamples=c["nvec"], tol=c["tol"], m_max=c["m_max"], z=s["v"])
        return s["x"]
    if kind == "solve":
        p.solve(s["v"], s["x"], nrhs=c["nvec"], tol=c["tol"], m_max=c["m_max"])
        return s["x"]
    if kind == "logdet":
        ld, _, q, _, _ = p.logdet(nprobes=c["nvec"], tol=c["tol"], m_max=c["m_max"], probes=s["v"])
        return {"logdet": ld, "q": q.astype(np.float32)}  # single-precision vectors: their quadratures carry that many digits
    if kind == "block":
        _, _, ld, _, q, _ = p.sample_logdet(s["x"], nsamples=c["nvec"], nprobes=c["nprobes"], tol=c["tol"],
                                            m_max=c["m_max"], z=s["v"], probes=s["probes"])
        return {"x": s["x"], "logdet": ld, "q": q.astype(np.float32)}
    if kind == "proposal":
        p.solve(s["b"], s["mean"], tol=c["tol"], m_max=c["m_max"])
        p.sample(s["x"], tol=c["tol"], m_max=c["m_max"], z=s["v"])
        return {"mean": s["mean"], "x": s["x"]}
    if kind == "sparse":
        p.sample(s["x"], nsamples=c["nvec"], tol=c["tol"], m_max=c["m_max"], z=s["v"])
        return s["x"]
    sv = s["server"]
    reqs = [sv.submit_sample(o, len(o), s["seed"] + i) for i, o in enumerate(s["out"])]
    last = sv.submit_logdet(c["probes"], s["seed"] + 100)
    while sv.step():
        pass
    got = [sv.poll(r) for r in reqs + [last]]
    return {"x": s["out"], "logdet": got[-1][2]}


# ------------------------------------------------------------------ what a pass cannot do without
def _steps(c):
    """Lanczos steps a pass takes, about: the square root of the condition number and the digits asked for."""
    kind = c["kind"]
    if kind in ("block", "serve", "solve") or c.get("precond") == "mirror":
        return 60
    if kind == "proposal":
        return 12
    if kind == "sparse":
        return 20
    low = {"const": CONST_K2, "smooth": 0.02, "uniform": 0.06}[c["field"]]
    cond = (low + (12 if c.get("nz") else 8)) / low
    return min(c["m_max"], int(0.45 * math.sqrt(cond) * math.log(2 / c["tol"])) + 4)


def work(case):
    c, kind = case, case["kind"]
    es = 8 if c.get("precision", "fp32") == "fp64" else 4
    if kind == "sparse":
        n, nv, m = c["side"] ** 2, c["nvec"], _steps(c)
        Q, F = _figure3(c["side"], c["droptol"], c["shift"])
        nnz = int(np.count_nonzero(Q)) + 2 * int(np.count_nonzero(F))
        # z in, x out, the basis written and read once, the matrices read once
        return {"bytes": nv * n * es * (2 + 2 * m) + nnz * 12, "flops": nv * m * (2.0 * nnz + 12 * n)}
    n = int(np.prod(_shape(c)))
    lg = math.log2(c["nx"])
    point = 26 if c.get("op") == "spde_squared" else (14 if c.get("nz") else 10)
    solve = 2 * 2.5 * lg + 10  # one B^{-1} in two dimensions, per cell: a transform each way along x, a recurrence along y
    if kind == "inv_sqrt":
        return {"bytes": 2 * c["nvec"] * n * es, "flops": c["nvec"] * n * solve}
    if kind == "apply":
        return {"bytes": 2 * c["nvec"] * n * es + 4 * n, "flops": c["nvec"] * n * point}
    m = _steps(c)
    pre = kind in ("solve", "block", "proposal", "serve") or c.get("precond") == "mirror"
    step = (2 * solve + 22) if pre else (point + 14)
    if kind == "logdet":
        return {"bytes": c["nvec"] * n * es + 4 * n, "flops": c["nvec"] * n * m * step}
    if kind == "block":
        return {"bytes": n * es * (c["nvec"] * (2 + 2 * m) + c["nprobes"]) + 4 * n,
                "flops": (c["nvec"] + c["nprobes"]) * n * m * step}
    if kind == "serve":
        nv = sum(int(k) for k in c["counts"].split(","))
        return {"bytes": n * es * nv * (1 + 2 * m) + 4 * n, "flops": (nv + c["probes"]) * n * m * step}
    nv = 2 if kind == "proposal" else c["nvec"]
    # z in, x out, the basis written and read once, kappa^2 read once
    return {"bytes": nv * n * es * (2 + 2 * m) + 4 * n, "flops": nv * n * m * step}


# ------------------------------------------------------------------ the same in 64 bits, in plain torch
def _lap(v, bc):
    """Graph Laplacian over the last dimensions of v [batch, ...]."""
    out = torch.zeros_like(v)
    for d in range(1, v.dim()):
        if bc == "periodic":
            out += 2 * v - torch.roll(v, 1, d) - torch.roll(v, -1, d)
            continue
        e = torch.diff(v, dim=d)
        k = v.shape[d]
        out.narrow(d, 0, k - 1).sub_(e)
        out.narrow(d, 1, k - 1).add_(e)
        if bc == "dirichlet":
            out.narrow(d, 0, 1).add_(v.narrow(d, 0, 1))
            out.narrow(d, k - 1, 1).add_(v.narrow(d, k - 1, 1))
    return out


def _dct(v):
    """DCT-II along the last axis (orthonormal), through one FFT."""
    N = v.shape[-1]
    u = torch.cat([v[..., ::2], v[..., 1::2].flip(-1)], -1)
    w = torch.exp(-1j * math.pi * torch.arange(N, device=v.device, dtype=torch.float64) / (2 * N))
    r = (torch.fft.fft(u) * w).real * math.sqrt(2.0 / N)
    r[..., 0] /= math.sqrt(2.0)
    return r


def _idct(C):
    N = C.shape[-1]
    C = C * math.sqrt(N / 2.0)
    C[..., 0] *= math.sqrt(2.0)
    rev = torch.cat([torch.zeros_like(C[..., :1]), C[..., 1:].flip(-1)], -1)
    w = torch.exp(1j * math.pi * torch.arange(N, device=C.device, dtype=torch.float64) / (2 * N))
    u = torch.fft.ifft((C - 1j * rev) * w).real
    out = torch.empty_like(C)
    out[..., ::2] = u[..., : (N + 1) // 2]
    out[..., 1::2] = u[..., (N + 1) // 2:].flip(-1)
    return out


def _inverse(shape, kind, k2):
    """v -> (k2 + L)^{-1} v with the Laplacian of the torus (circulant) or of the reflected grid (mirror)."""
    step = 2 if kind == "circulant" else 1
    lam = k2
    for d, s in enumerate(shape):
        a = torch.arange(s, device="cuda", dtype=torch.float64) * (math.pi * step / s)
        lam = lam + (4 * torch.sin(a / 2) ** 2).reshape([-1 if e == d else 1 for e in range(len(shape))])
    if kind == "circulant":
        return lambda v: torch.fft.ifft2(torch.fft.fft2(v) / lam).real
    return lambda v: _idct(_idct((_dct(_dct(v).transpose(1, 2)) / lam.t())).transpose(1, 2))


def _lanczos(op, z, outs, cap=400, eps=1e-13):
    """For each vector of z [b, n]: ||z|| V f(T) e_1 for f = t^{-1/2} ("sample") or 1/t ("solve"), or ||z||^2 e_1' log T e_1 ("log")."""
    b, n = z.shape
    norm = z.norm(dim=1, keepdim=True)
    V, al, be = [z / norm], [], []
    while True:
        v = V[-1]
        w = op(v)
        al.append((w * v).sum(1))
        B = torch.stack(V, 1)
        for _ in range(2):
            w = w - torch.einsum("bjn,bj->bn", B, torch.einsum("bjn,bn->bj", B, w))
        del B
        be.append(w.norm(dim=1))
        m = len(al)
        if m % 8 == 0 or m >= cap or m >= n:
            T = torch.diag_embed(torch.stack(al, 1))
            if m > 1:
                o = torch.stack(be[:-1], 1)
                T = T + torch.diag_embed(o, 1) + torch.diag_embed(o, -1)
            lam, U = torch.linalg.eigh(T)
            f = {"sample": lambda t: t.rsqrt(), "solve": lambda t: 1 / t, "log": torch.log}[outs](lam)
            y = torch.einsum("bij,bj->bi", U, f * U[:, 0])
            tail = y[:, -2:].abs().amax(1) / y.norm(dim=1)
            if m >= cap or m >= n or float(tail.max()) < eps:
                if outs == "log":
                    return norm[:, 0] ** 2 * y[:, 0]
                return norm * torch.einsum("bjn,bj->bn", torch.stack(V, 1), y)
        V.append(w / be[-1][:, None])


def _batched(op, z, outs, each):
    return torch.cat([_lanczos(op, z[i:i + each].double(), outs) for i in range(0, len(z), each)])


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "serve":
        return None  # the server draws its own noise
    if kind == "sparse":
        Q, F = (torch.from_numpy(a).cuda() for a in _figure3(c["side"], c["droptol"], c["shift"]))
        z = _randn((c["nvec"], len(Q)), seed, 2, torch.float64)
        A = torch.linalg.solve_triangular(F, torch.linalg.solve_triangular(F, Q, upper=False).t(), upper=False)
        lam, U = torch.linalg.eigh((A + A.t()) / 2)
        u = U @ (lam.rsqrt()[:, None] * (U.t() @ z.t()))
        return torch.linalg.solve_triangular(F.t(), u, upper=True).t().contiguous()
    shape = _shape(c)
    n = int(np.prod(shape))
    grid = lambda v: v.reshape((-1,) + shape)  # noqa: E731
    flat = lambda v: v.reshape(v.shape[0], -1)  # noqa: E731
    each = max(1, int(6e9 / (8.0 * n * 150)))
    if kind == "inv_sqrt":
        return flat(_inverse(shape, c["precond"], MEAN_K2)(grid(_noise(c, seed, c["nvec"]).double())))
    if kind == "proposal":
        m = _lgcp(c, seed)
        P, D = _inverse(shape, "circulant", m["kc2"]), m["d"].double()
        op = lambda v: v + flat(P(D * P(grid(v))))  # noqa: E731
        z, b = _noise(c, seed, 1), m["grad"].to(torch.float64 if c["precision"] == "fp64" else torch.float32)
        start = flat(P(grid(b[None].double())))
        mean = flat(P(grid(_lanczos(op, start, "solve"))))[0] / m["tau"]
        x = flat(P(grid(_lanczos(op, z.double(), "sample")))) / math.sqrt(m["tau"])
        return {"mean": mean, "x": x}
    bc = c.get("bc", "neumann")
    k2 = _field(c, seed)
    k2 = torch.full(shape, CONST_K2, device="cuda", dtype=torch.float64) if k2 is None else k2.double()
    B = lambda v: k2 * v + _lap(v, bc)  # noqa: E731
    squared = c.get("op", "spde_squared") == "spde_squared"
    Q = (lambda v: B(B(v))) if squared else B
    if kind == "apply":
        return flat(Q(grid(_noise(c, seed, c["nvec"]).double())))
    nv = c["nvec"] + c.get("nprobes", 0)
    steps = 100 if squared else 1.5 * _steps(c)
    if nv * n * steps * (steps + 120) > 4e12:
        return None  # over the time an exact answer may take
    pre = kind in ("solve", "block") or c.get("precond") == "mirror"
    if not pre:
        op = lambda v: flat(Q(grid(v)))  # noqa: E731
        if kind == "logdet":
            q = _batched(op, _probes(c, seed, c["nvec"]), "log", each)
            return {"logdet": float(q.mean()), "q": q}
        return _batched(op, _noise(c, seed, c["nvec"]), "sample", each)
    kbar = float(torch.exp(torch.log(k2).mean()))
    P = _inverse(shape, "mirror", kbar)
    op = lambda v: flat(P(Q(P(grid(v)))))  # noqa: E731
    if kind == "solve":
        b = _noise(c, seed, c["nvec"]).double()
        return flat(P(grid(_batched(op, flat(P(grid(b))), "solve", each))))
    lam = torch.zeros((), device="cuda", dtype=torch.float64) + kbar
    for d, s in enumerate(shape):
        a = torch.arange(s, device="cuda", dtype=torch.float64) * (math.pi / s)
        lam = lam + (4 * torch.sin(a / 2) ** 2).reshape([-1 if e == d else 1 for e in range(len(shape))])
    logdet_M = float(2 * torch.log(lam).sum())
    if kind == "logdet":
        q = _batched(op, _probes(c, seed, c["nvec"]), "log", each)
        return {"logdet": float(q.mean()) + logdet_M, "q": q}
    x = flat(P(grid(_batched(op, _noise(c, seed, c["nvec"]), "sample", each)))) if kind in ("sample", "block") else None
    if kind == "sample":
        return x
    q = _batched(op, _probes(c, seed, c["nprobes"]), "log", each)
    return {"x": x, "logdet": float(q.mean()) + logdet_M, "q": q}
