"""Columns that the mixed warp kernels hand to the FP64 kernel with I_j already
decided (A without the rows of I_j is too ill-conditioned for FP32, T is not):
the FP64 kernel takes I_j from the mixed kernel and the host's walk of V's
levels passes the column before that kernel has run.  Factors against the
oracle, and the first apply (enqueued right behind) against the oracle's
preconditioner, real and complex, both triangular rules.
Tolerances are those of the parity suites and of the streamed-schedule suite."""
import gc

import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
from tests._parity import assert_parity, compare, host_factors
from tests._problems import pattern_from_sets
from workloads import CSC

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def nearly_parallel(n, pairs, cplx, seed):
    """A band with, for every a of pairs, column a + 1 equal to column a up to
    1e-3 and a diagonal entry."""
    rng = np.random.default_rng(seed)
    M = np.zeros((n, n), np.complex128 if cplx else np.float64)

    def draw(size):
        return rng.standard_normal(size) + (1j * rng.standard_normal(size) if cplx else 0.0)

    for j in range(n):
        rows = np.arange(max(0, j - 5), min(n, j + 6))
        M[rows, j] = draw(rows.size)
        M[j, j] += 12.0
    for a in pairs:
        rows = np.arange(max(0, a - 5), min(n, a + 6))
        M[a, a] -= 8.0
        M[:, a + 1] = M[:, a]
        M[rows, a + 1] += 1e-3 * draw(rows.size)
        M[a + 1, a + 1] += 8.0
    return CSC.from_scipy(sp.csc_matrix(M))


def problem(n, cplx, rule):
    pairs = [8, 18] + list(range(40, n - 8, 12))
    A = nearly_parallel(n, pairs, cplx, 3)
    if rule == O.RULE_UPPER:
        sets = [range(j - 2, j + 1) if j - 1 in pairs else [j] for j in range(n)]
    else:
        sets = [range(j, j + 3) if j in pairs else [j] for j in range(n)]
    budget = np.array([2 if len(s) == 3 else 1 for s in sets], np.int32)
    return pairs, A, pattern_from_sets(n, sets), budget


@pytest.mark.parametrize("rule", [O.RULE_UPPER, O.RULE_LOWER])
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n", [33, 400])
def test_decided_columns(n, cplx, rule):
    from paper_1208_3573_gb300 import diaf
    diaf.lib()
    gc.collect()  # no earlier factors hold the host copy of V's structure
    pairs, A, PW, budget = problem(n, cplx, rule)
    o = O.factor(A, PW, rule, budget, alg="S")
    x = np.random.default_rng(5).standard_normal(n) + (1j if cplx else 0.0)
    xd = torch.from_numpy(x).cuda()
    dA, dP = diaf.DeviceCSC.from_host(A), diaf.DeviceCSC.from_host(PW)
    dB = torch.from_numpy(budget).cuda()
    s0, c0 = diaf.apply_prep_counts()
    F = diaf.factor(dA, dP, rule, dB, alg="S", prec="mixed32")
    y = F.apply(xd)  # at once: the walk runs during the numeric pass
    F.sync()
    s1, c1 = diaf.apply_prep_counts()
    assert (s1 - s0, c1 - c0) == (1, 0)
    assert sum(F.fallbacks()) == len(pairs)
    assert_parity(compare(host_factors(F), o, A, PW, "S", rtol_res=1e-4, vec_tol=1e-6, mixed=True, floor_rel=1e-10))
    yr = O.Preconditioner(o.W_csc(), o.V_csc())(x)
    assert np.linalg.norm(y.cpu().numpy() - yr) <= 1e-8 * np.linalg.norm(yr)
    F.close()
