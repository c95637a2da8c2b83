"""Columns of A whose entries leave the range of FP32 squares beside ordinary
ones: rows of a Dirichlet condition imposed by a penalty of 1e22 or 1e30 on the
diagonal, and columns scaled by 1e-22 (mixed precision).  Every tile that holds
such a column has to go to the FP64 kernel as a whole -- one lane of a warp that
decides otherwise would leave the others in another branch -- so its W, V and
I_j are the FP64 set-up's bit for bit; every other column is bit for bit what it
is without them."""
import numpy as np
import pytest

import oracle as O
from tests._parity import host_factors
from tests.test_gpu_parity import run_gpu
from workloads import CSC, make_workload

pytestmark = pytest.mark.gpu

PROBLEMS = ["convdiff48_A2", "helmholtz40", "lognormal16", "powerlaw6k"]  # every mixed kernel's tiles


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import build, diaf
    build.build()
    return diaf


def special_columns(w):
    """Lone columns, and one that is the first and one that is the last of some tile."""
    rng = np.random.default_rng(3)
    c = set(rng.choice(w.n, 6, replace=False).tolist())
    mid = w.n // 2 + 5
    J = w.PW.rowidx[w.PW.colptr[mid]:w.PW.colptr[mid + 1]]
    return np.asarray(sorted(c | {int(J[0])})), np.asarray([int(J[-1])])


def with_special(A, cols, kind):
    vals = A.vals.copy()
    for c in cols:
        s = slice(A.colptr[c], A.colptr[c + 1])
        if kind < 1.0:
            vals[s] *= kind
        else:
            vals[s][A.rowidx[s] == c] = kind
    return CSC(A.n, A.colptr, A.rowidx, vals)


def column(g, which, j):
    cp, ri, v = (g["Wcp"], g["Wri"], g["Wv"]) if which == "W" else (g["Vcp"], g["Vri"], g["Vv"])
    return ri[cp[j]:cp[j + 1]].tolist(), v[cp[j]:cp[j + 1]].tobytes()


@pytest.mark.parametrize("alg", ["S", "Q"])
@pytest.mark.parametrize("kind", [1e22, 1e30, 1e-22])
@pytest.mark.parametrize("name", PROBLEMS)
def test_columns_out_of_range(D, name, kind, alg):
    w = make_workload(name)
    args = dict(alg=alg, tie_tol=w.tie_tol)
    plain = host_factors(run_gpu(D, w.A, w.PW, w.vrule, w.budget, prec="mixed32", **args))
    for cols in special_columns(w):
        A = with_special(w.A, cols, kind)
        g = host_factors(run_gpu(D, A, w.PW, w.vrule, w.budget, prec="mixed32", **args))
        f = host_factors(run_gpu(D, A, w.PW, w.vrule, w.budget, prec="fp64", **args))
        hit = np.zeros(w.n, bool)
        for j in range(w.n):
            hit[j] = np.isin(cols, w.PW.rowidx[w.PW.colptr[j]:w.PW.colptr[j + 1]]).any()
        assert 0 < hit.sum() < w.n
        assert (g["flags"][hit] & 64).all()
        assert np.array_equal(g["Vcp"], f["Vcp"])
        for j in range(w.n):
            ref = f if hit[j] else plain
            for which in "WV":
                assert column(g, which, j) == column(ref, which, j), (j, which, bool(hit[j]))
