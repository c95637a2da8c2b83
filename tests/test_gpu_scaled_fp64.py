"""FP64 DIAF-S in other units: every scalar of the direct form is of the tile's
precision, so 2^e A takes the same steps as A as far as FP64 reaches, and most
columns of W keep every bit (a column that went to the Jacobi instead would
keep hardly any)."""
import numpy as np
import pytest

from tests._parity import host_factors
from tests.test_gpu_parity import run_gpu
from workloads import CSC, make_workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import build, diaf
    build.build()
    return diaf


@pytest.mark.parametrize("log2c", [-200, -70, 70, 200])
@pytest.mark.parametrize("name", ["convdiff48_A2", "lognormal16"])
def test_same_steps(D, name, log2c):
    w = make_workload(name)
    A = CSC(w.A.n, w.A.colptr, w.A.rowidx, w.A.vals * 2.0 ** log2c)
    g, s = (host_factors(run_gpu(D, M, w.PW, w.vrule, w.budget, alg="S", prec="fp64", tie_tol=w.tie_tol))
            for M in (w.A, A))
    same = [np.array_equal(g["Wv"][a:b], s["Wv"][a:b]) for a, b in zip(g["Wcp"], g["Wcp"][1:])]
    assert np.mean(same) > 0.5
