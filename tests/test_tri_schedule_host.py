"""The merged levels of the triangular solves (tri_schedule.h, compiled for the host): every coefficient is the exact one
rounded once, and no merge loses more digits than its stated growth.  No GPU."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from oracle import sparse as osp
from paper_1312_1476_gb300 import _build, inputs

SOURCE = r"""
#include "tri_schedule.h"
using namespace gmrf;
static TriHost h;
extern "C" int build(int n, const int* ptr, const int* col, const double* val, const double* dg, int forward) {
  const std::vector<int> p(ptr, ptr + n + 1), c(col, col + ptr[n]);
  const std::vector<double> v(val, val + ptr[n]), d(dg, dg + n);
  std::vector<int> rows, lptr;
  levels(n, p, c, forward != 0, rows, lptr);
  tri_schedule(n, rows, lptr, p, c, v, d, forward != 0, forward ? 2 * n : 0, n, h);
  return (int)h.rec.size() / 8;
}
extern "C" const int* recs() { return h.rec.data(); }
extern "C" const int* row() { return h.row.data(); }
extern "C" const int* col() { return h.col.data(); }
extern "C" const double* val() { return h.val.data(); }
"""
GROWTH = 10  # kGrowth


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("tri")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", _build.CSRC, str(d / "t.cpp"), "-o",
                    str(d / "t.so")], check=True)
    so = ctypes.CDLL(str(d / "t.so"))
    for name in ("recs", "row", "col"):
        getattr(so, name).restype = ctypes.POINTER(ctypes.c_int)
    so.val.restype = ctypes.POINTER(ctypes.c_double)
    return so


def _schedule(lib, F, forward):
    """[(rows, {row: {position: coefficient}}) of each merged level] of F x = b (forward) or F' x = b, and the rows' entries."""
    n = F.shape[0]
    T = (F if forward else F.T).tocsr()
    T.sort_indices()
    off = [[(int(c), float(v)) for c, v in zip(T.indices[T.indptr[i]:T.indptr[i + 1]], T.data[T.indptr[i]:T.indptr[i + 1]])
            if c != i] for i in range(n)]
    dg = np.ascontiguousarray(F.diagonal())
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in off])]).astype(np.int32)
    col = np.array([c for r in off for c, _ in r] or [0], dtype=np.int32)
    val = np.array([v for r in off for _, v in r] or [0.0])
    rounds = lib.build(n, *(a.ctypes.data_as(ctypes.c_void_p) for a in (ptr, col, val, dg)), int(forward))
    R = np.ctypeslib.as_array(lib.recs(), (rounds, 8))
    out, level = [], {}
    for at, slots, lanes, lg, first, count, last, _ in R.tolist():
        C = np.ctypeslib.as_array(lib.col(), (at + slots * lanes,))[at:].reshape(slots, lanes)
        V = np.ctypeslib.as_array(lib.val(), (at + slots * lanes,))[at:].reshape(slots, lanes)
        for g in range(count):
            c, v = C[:, g << lg:(g + 1) << lg].ravel(), V[:, g << lg:(g + 1) << lg].ravel()
            level[lib.row()[first + g]] = {int(a): float(b) for a, b in zip(c, v) if a >= 0}
        if last:
            out.append(level)
            level = {}
    assert not level and sum(len(x) for x in out) == n
    return out, off, dg


def _factor(kind, n=96):
    rng = np.random.default_rng(7)
    if kind == "ichol":
        return osp.ichol(osp.csr(*inputs.random_sparse_spd(9, 7, seed=13, squared=True)), droptol=1e-4, shift=0.05).tocsr()
    # far from diagonally dominant, and with rows of very different sizes
    F = np.tril(np.triu(rng.standard_normal((n, n)) * 3, -3), -1) + np.diag(rng.uniform(0.5, 2.0, n))
    if kind == "scaled":
        F = np.exp2(rng.integers(-30, 30, n))[:, None] * F
    r, c = np.nonzero(F)
    return osp.csr(np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]), c, F[r, c]).tocsr()


@pytest.mark.parametrize("forward", [True, False], ids=["forward", "backward"])
@pytest.mark.parametrize("kind", ["ichol", "growing", "scaled"])
def test_coefficients_are_rounded_once(lib, kind, forward):
    F = _factor(kind)
    n = F.shape[0]
    levels, off, dg = _schedule(lib, F, forward)
    b0 = 2 * n if forward else 0
    merged = 0
    for level in levels:
        exact, paths = {}, {}
        for i in sorted(level, reverse=not forward):
            e, a = {b0 + i: Fraction(1)}, {b0 + i: Fraction(1)}
            for k, v in off[i]:
                src = exact[k] if k in level else {n + k: Fraction(1)}
                mag = paths[k] if k in level else src
                for t in src:
                    e[t] = e.get(t, 0) - Fraction(v) * src[t]
                    a[t] = a.get(t, 0) + abs(Fraction(v)) * mag[t]
            d = Fraction(float(dg[i]))
            exact[i], paths[i] = {t: c / d for t, c in e.items()}, {t: c / d for t, c in a.items()}
            assert set(level[i]) == set(exact[i])
            merged += any(k in level for k, _ in off[i])
            for t, c in level[i].items():
                # half an ulp, and twice the working digits less a few for what cancels between the paths
                assert abs(Fraction(c) - exact[i][t]) <= abs(exact[i][t]) * Fraction(1, 2 ** 53) + paths[i][t] / 2 ** 95
    assert merged  # something was merged at all


@pytest.mark.parametrize("precision", [np.float32, np.float64])
@pytest.mark.parametrize("forward", [True, False], ids=["forward", "backward"])
@pytest.mark.parametrize("kind", ["ichol", "growing", "scaled"])
def test_residual_of_a_merged_solve(lib, kind, forward, precision):
    """b = F x with |x_k| = omega_k.  A row of L entries is off by at most (L + 2) u sum |c s| (its coefficients rounded
    once more to the precision, its products, its sum), the sum at most GROWTH times the row's own substitution's
    while sources are of the sizes that the rule assumes, mu times that otherwise; the residual adds F times that."""
    F = _factor(kind)
    n = F.shape[0]
    levels, off, dg = _schedule(lib, F, forward)
    u = float(np.finfo(precision).eps) / 2
    omega = np.ones(n) if forward else 1 / dg
    size = np.array([dg[i] * omega[i] + sum(abs(v) * omega[k] for k, v in off[i]) for i in range(n)])
    sign = np.where(np.random.default_rng(3).random(n) < 0.5, -1.0, 1.0)
    b = np.array([precision(sum((Fraction(v) * Fraction(float(sign[k] * omega[k])) for k, v in off[i]),
                                Fraction(float(dg[i])) * Fraction(float(sign[i] * omega[i])))) for i in range(n)], precision)
    sm = np.zeros(3 * n, precision)
    b0 = 2 * n if forward else 0
    sm[b0:b0 + n] = b
    longest = 0
    for level in levels:
        new = {}
        for i, row in level.items():
            longest = max(longest, len(row))
            acc = precision(0)
            for t, c in row.items():
                acc = precision(acc + precision(c) * sm[t])
            new[i] = acc
        for i, v in new.items():
            sm[n + i] = v
    x = sm[n:2 * n]
    mu = max(1.0, float(np.max(np.abs(x) / omega)))
    gamma = (longest + 3) * u
    gamma = gamma / (1 - gamma)
    where = {i: s for s, level in enumerate(levels) for i in level}
    for i in range(n):
        res = Fraction(float(b[i])) - Fraction(float(dg[i])) * Fraction(float(x[i])) - \
            sum(Fraction(v) * Fraction(float(x[k])) for k, v in off[i])
        spread = size[i] + sum(abs(v) * size[k] / dg[k] for k, v in off[i] if where[k] == where[i])
        assert abs(float(res)) <= 1.01 * gamma * GROWTH * mu * spread
