"""DIAF-S columns of the large-tile mixed-precision kernel (one CTA per
column): sparse tiles at the edges of its capacity (k_j = 1 to 64, m_j up to
1024), the products over the gathered entries, two words of column mask per
row, odd k_j in the pairing of the rotations, stored zeros and a column whose
only nonzero lies in a row of I_j, against the oracle.  Tolerances are those of
the parity suites."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
from tests._parity import assert_parity, compare, host_factors
from tests._problems import pattern_from_sets
from tests.test_gpu_parity import run_gpu
from workloads import CSC

pytestmark = pytest.mark.gpu


def scattered(n, per, seed, big, zeros=False):
    """`per` entries per column at random rows, a diagonal of about 4 to 8;
    with zeros, half of the off-diagonal entries are stored zeros and column
    b + 1 of every b in big is one entry in row b (a zero column outside I_b)."""
    rng = np.random.default_rng(seed)
    ci, ri, va = [], [], []
    for j in range(n):
        rows = np.unique(np.append(rng.choice(n, per - 1, replace=False), j))
        v = rng.standard_normal(rows.size)
        if zeros:
            v[rng.random(rows.size) < 0.5] = 0.0
        v[rows == j] = rng.uniform(4.0, 8.0)
        if zeros and j - 1 in big:
            rows, v = np.unique(np.append(rows, j - 1)), None
            v = np.where(rows == j - 1, 1.5, 0.0)
        ri.append(rows)
        va.append(v)
        ci.append(rows.size)
    colptr = np.concatenate([[0], np.cumsum(ci)])
    return CSC.from_scipy(sp.csc_matrix((np.concatenate(va), np.concatenate(ri), colptr), (n, n)))


@pytest.mark.parametrize("k,per,zeros", [(1, 400, False), (2, 500, False), (17, 20, False), (32, 31, False),
                                         (33, 9, False), (33, 9, True), (63, 3, False), (63, 15, True),
                                         (64, 15, False)])
def test_large_sparse_tiles(k, per, zeros):
    n = 4000
    big = [100, 101 + k, 900, 1700, 2500, 3300]
    A = scattered(n, per, k + per, set(big), zeros)
    PW = pattern_from_sets(n, [range(j, j + k) if j in big else [j] for j in range(n)])
    budget = np.where(np.isin(np.arange(n), big), 5, 1).astype(np.int32)
    from paper_1208_3573_gb300 import diaf
    diaf.lib()
    F = run_gpu(diaf, A, PW, O.RULE_UPPER, budget, alg="S", prec="mixed32")
    o = O.factor(A, PW, O.RULE_UPPER, budget, alg="S")
    assert_parity(compare(host_factors(F), o, A, PW, "S", rtol_res=1e-4, vec_tol=1e-6, mixed=True, floor_rel=1e-10))
