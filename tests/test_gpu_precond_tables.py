"""A preconditioned problem holds the tables that its kernels read, and no others."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

USED_MEM_CURRENT = 7  # cudaMemPoolAttrUsedMemCurrent


def _pool_bytes():
    from paper_1312_1476_gb300 import gmrf  # noqa: F401  (loads the runtime)
    rt = ctypes.CDLL("libcudart.so.13")
    torch.cuda.synchronize()
    pool, used = ctypes.c_void_p(), ctypes.c_uint64()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    assert rt.cudaMemPoolGetAttribute(pool, USED_MEM_CURRENT, ctypes.byref(used)) == 0
    return used.value


@pytest.mark.parametrize("kind,bc", [("mirror", "neumann"), ("circulant", "periodic")])
@pytest.mark.parametrize("precision,size", [("fp32", 4), ("fp64", 8)])
def test_squared_operator_holds_its_line_tables_only(kind, bc, precision, size):
    from paper_1312_1476_gb300 import gmrf
    nx = 1024
    with gmrf.Problem((nx, nx), bc, "spde_squared", kappa2_const=0.1, precond=kind, precision=precision):
        pass  # what the first problem of a process sets up
    before = _pool_bytes()
    with gmrf.Problem((nx, nx), bc, "spde_squared", kappa2_const=0.1, precond=kind, precision=precision):
        held = _pool_bytes() - before
    # reals: 7 twiddles at each of the strides 8 and 64 of a 512-point transform, 4 or 2 a pair, 8 a column
    tables = 2 * 7 * (8 + 64) + (4 if kind == "mirror" else 2) * nx // 4 + 8 * nx
    assert 0 < held <= tables * size + 3 * 512  # three allocations
