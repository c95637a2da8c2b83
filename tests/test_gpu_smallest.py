"""DIAF-S columns whose smallest singular vector comes from the direct path of
the warp kernels (Gram matrix, swept inverses, corrections): tile widths at
the edges of the kernels' capacities, every precision and value type, tiles
that fall apart into unconnected columns (exact zeros in w, v_jj = 0), equal
singular values and an ill-conditioned tile (the Jacobi path), against the
oracle.  Tolerances are those of the parity suites."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
from tests._parity import assert_parity, compare, host_factors
from tests._problems import pattern_from_sets
from tests.test_gpu_parity import run_gpu
from workloads import CSC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import diaf
    diaf.lib()
    return diaf


def banded(n, seed, cplx, diag=6.0, scale=0.0, bands=4):
    rng = np.random.default_rng(seed)
    M = sp.diags([rng.standard_normal(n - abs(d)) + (diag if d == 0 else 0.0) for d in range(-bands, bands + 1)],
                 range(-bands, bands + 1)).tocsc()
    if cplx:
        M = M.astype(np.complex128)
        M.data = M.data * np.exp(1j * rng.uniform(0, 2 * np.pi, M.data.size))
    if scale:
        M = (M @ sp.diags(10.0 ** rng.uniform(-scale, scale, n))).tocsc()
    return CSC.from_scipy(M)


def window(n, k):
    return pattern_from_sets(n, [range(max(0, min(j - k // 2, n - k)), max(0, min(j - k // 2, n - k)) + k)
                                 for j in range(n)])


def check(D, A, PW, prec):
    budget = np.full(A.n, 2, np.int32)
    g = host_factors(run_gpu(D, A, PW, O.RULE_UPPER, budget, alg="S", prec=prec))
    o = O.factor(A, PW, O.RULE_UPPER, budget, alg="S")
    if prec == "fp64":
        assert_parity(compare(g, o, A, PW, "S"))
    else:
        assert_parity(compare(g, o, A, PW, "S", rtol_res=1e-4, vec_tol=1e-6, mixed=True, floor_rel=1e-10))


@pytest.mark.parametrize("prec", ["fp64", "mixed32"])
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("k", [1, 2, 3, 9, 15, 16, 17, 25, 31, 32])
def test_tile_widths(D, k, cplx, prec):
    A = banded(70, k, cplx, scale=1.0 if k % 2 else 0.0)
    check(D, A, window(70, k), prec)


@pytest.mark.parametrize("prec", ["fp64", "mixed32"])
@pytest.mark.parametrize("kind", ["unconnected", "equal", "ill"])
def test_special_tiles(D, kind, prec):
    n = 60
    if kind == "unconnected":  # every second off-diagonal pair missing: tiles of 2 x 2 blocks
        M = banded(n, 5, False, bands=1).to_scipy().tolil()
        for i in range(1, n - 1, 2):
            M[i, i + 1] = M[i + 1, i] = 0.0
        A = CSC.from_scipy(sp.csc_matrix(M.tocsc()))
        A = CSC.from_scipy(sp.csc_matrix((A.vals[A.vals != 0], A.rowidx[A.vals != 0],
                                          np.concatenate([[0], np.cumsum([np.count_nonzero(
                                              A.vals[A.colptr[j]:A.colptr[j + 1]]) for j in range(n)])])), (n, n)))
    elif kind == "equal":  # orthogonal columns of equal norm
        A = CSC.from_scipy(sp.csc_matrix(2.0 * sp.identity(n, format="csc")))
    else:  # nearly parallel columns
        M = banded(n, 7, False, bands=1).to_scipy()
        A = CSC.from_scipy(sp.csc_matrix(M @ (sp.identity(n) + sp.diags([np.full(n - 1, 50.0)], [1]))))
    check(D, A, window(n, 8), prec)
