"""A context that cannot place the clusters of the small 2-D grids (one limited to a few SMs): the one-step kernel serves
them, with the same bits.  A child process runs with a fake cudaOccupancyMaxActiveClusters that finds no room."""
import json
import os
import subprocess
import sys

import pytest

from paper_1312_1476_gb300 import _build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CALLS = r"""
import json, sys
import torch
from paper_1312_1476_gb300 import gmrf
out = []
for precision, dtype in (("fp64", torch.float64), ("fp32", torch.float32)):
    for bc in ("periodic", "neumann", "dirichlet"):
        for shape in ((9, 33), (64, 64)):
            n = shape[0] * shape[1]
            z = torch.randn(2, n, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda", dtype=dtype)
            x, y = torch.empty_like(z), torch.empty_like(z)
            with gmrf.Problem(shape, bc, "shifted_laplacian", kappa2_const=0.3, precision=precision) as p:
                gmrf.trace_reset()
                rc, info = p.sample(x, nsamples=2, z=z, tol=1e-5, m_max=80)
                steps = gmrf.trace_query("stencil_step")[1]
                p.solve(z, y, nrhs=2, tol=1e-5, m_max=80)
            out.append([rc, info[0].m_used, info[1].m_used, steps > 4, x.tolist(), y.tolist()])
json.dump(out, sys.stdout)
"""

FAKE = 'extern "C" int cudaOccupancyMaxActiveClusters(int* n, const void*, const void*) { *n = 0; return %d; }\n'


def _run(**env):
    r = subprocess.run([sys.executable, "-c", CALLS], cwd=_build.ROOT, env=dict(os.environ, **env), capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout)


@pytest.mark.parametrize("code", [0, 1], ids=["no room", "query fails"])
def test_one_step_kernel_serves(tmp_path, code):
    src, so = tmp_path / "fake.cpp", tmp_path / "fake.so"
    src.write_text(FAKE % code)
    subprocess.run(["g++", "-shared", "-fPIC", str(src), "-o", str(so)], check=True)
    plain, without = _run(), _run(LD_PRELOAD=str(so))
    for a, b in zip(plain, without):
        assert a[0] == b[0] == 0 and a[1:3] == b[1:3] and a[4:] == b[4:]
        assert not a[3] and b[3]  # all steps in one launch, and a launch a step
