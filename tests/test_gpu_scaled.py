"""A in other units: c A for c a power of two has the W of A, c times its V
and residuals (DIAF-S), or 1 / c times its W (DIAF-Q), with the same I_j and
flags, in both precisions and on every kernel's tiles.  Multiplying by a power of
two commutes with every rounding, so nothing but overflow and underflow can
tell c A from A: the same columns stay in mixed precision and the bound below
(1e-9 of the column) is for approximate reciprocals only."""
import numpy as np
import pytest

from tests._parity import host_factors
from tests.test_gpu_parity import run_gpu
from workloads import CSC, make_workload

pytestmark = pytest.mark.gpu

PROBLEMS = ["convdiff48_A2", "helmholtz40", "lognormal16", "powerlaw6k"]


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import build, diaf
    build.build()
    return diaf


def column_error(cp, x, y):
    """Per column: the largest difference over the largest entry of y."""
    col = np.repeat(np.arange(cp.size - 1), np.diff(cp))
    d, s = np.zeros(cp.size - 1), np.zeros(cp.size - 1)
    np.maximum.at(d, col, np.abs(x - y))
    np.maximum.at(s, col, np.abs(y))
    return d / np.maximum(s, 1e-300)


@pytest.mark.parametrize("prec", ["mixed32", "fp64"])
@pytest.mark.parametrize("alg", ["S", "Q"])
@pytest.mark.parametrize("log2c", [-200, -40, -25, 30, 40, 200])
@pytest.mark.parametrize("name", PROBLEMS)
def test_units(D, name, log2c, alg, prec):
    w = make_workload(name)
    c = 2.0 ** log2c
    A = CSC(w.A.n, w.A.colptr, w.A.rowidx, w.A.vals * c)
    args = dict(alg=alg, prec=prec, tie_tol=w.tie_tol)
    g = host_factors(run_gpu(D, w.A, w.PW, w.vrule, w.budget, **args))
    s = host_factors(run_gpu(D, A, w.PW, w.vrule, w.budget, **args))
    assert np.array_equal(s["Vcp"], g["Vcp"]) and np.array_equal(s["Vri"], g["Vri"])
    assert np.array_equal(s["flags"], g["flags"])
    cw, cv = (1.0, c) if alg == "S" else (1.0 / c, 1.0)
    unique = (g["flags"] & (1 | 2 | 32)) == 0  # not rank deficient, degenerate or empty
    for cp, key, f in ((g["Wcp"], "Wv", cw), (g["Vcp"], "Vv", cv)):
        err = column_error(cp, s[key] / f, g[key])
        assert err[unique].max() <= 1e-9, (key, int(np.argmax(np.where(unique, err, 0))))
    assert np.allclose(s["res"] / cv, g["res"], rtol=1e-9, atol=1e-12 * np.abs(w.A.vals).max() if alg == "S" else 1e-12)
