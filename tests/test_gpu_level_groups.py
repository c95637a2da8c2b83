"""The level solve's packed form (up to four off-diagonal entries per row) at
the edges of its rules: groups at and beyond a block's rows, one row per
level, rows whose merged entries do not fit, entries further back than the
shared-memory window, more level pointers than shared memory holds, five
entries per row (the general form), real and complex, upper and lower.

W is diagonal and V's pattern is A's, so V is A up to signs; y = W V^-1 x is
compared with a sparse direct solve.  A is column diagonally dominant with a
factor of 2, so ||V^-1|| ||V|| <= 4 in the 1-norm and the forward error is
below 4 (entries + 2) n_levels eps < 1e-11 for every case here."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spl

from tests._problems import pattern_from_matrix
from workloads import CSC

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import build, diaf
    build.build()
    return diaf


def layered(widths, parents, seed, far=False):
    """Strictly upper pattern (row i depends on columns j > i) with the given
    level widths; every row has `parents` entries in the next level(s)."""
    rng = np.random.default_rng(seed)
    n = int(np.sum(widths))
    ends = np.cumsum(widths)  # level l holds the rows n - ends[l] .. n - ends[l - 1] - 1
    rows, cols = [], []
    for l in range(1, len(widths)):
        for i in range(n - ends[l], n - ends[l - 1]):
            lo, hi = n - ends[l - 1], n - (ends[l - 2] if l > 1 else 0)
            c = {int(rng.integers(lo, hi))}  # one entry in the level before: the level is exact
            while len(c) < min(parents, n - lo):
                c.add(int(rng.integers(lo, n if far else min(n, hi + widths[max(l - 2, 0)]))))
            rows += [i] * len(c)
            cols += sorted(c)
    return n, np.asarray(rows, int), np.asarray(cols, int)


CASES = {
    "groups_1024": ([256] * 10, 2, False),
    "groups_beyond_block": ([257] * 9 + [1500, 3], 2, False),
    "groups_small": ([3, 1, 7, 2, 5, 1, 1], 3, False),
    "one_row_levels": ([1] * 300, 1, False),
    "merge_full": ([40] * 24, 4, True),
    "beyond_window": ([9000, 9000, 500, 500, 500], 2, True),
    "pointers_beyond_smem": ([1] * 9001, 1, False),
    "pointers_beyond_smem_ungrouped": ([1] * 33000, 1, False),
    "five_entries": ([50] * 12, 5, True),
    "single": ([1], 0, False),
}


@pytest.mark.parametrize("lower", [False, True])
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("case", list(CASES))
def test_packed_level_solve(D, case, cplx, lower):
    widths, parents, far = CASES[case]
    n, rows, cols = layered(widths, parents, 3, far)
    if lower:
        rows, cols = n - 1 - rows, n - 1 - cols
    rng = np.random.default_rng(7)
    v = rng.uniform(0.5, 1.0, rows.size) * rng.choice([-1.0, 1.0], rows.size)
    if cplx:
        v = v * np.exp(1j * rng.uniform(0, 2 * np.pi, rows.size))
    dom = 2.0 * np.bincount(cols, np.abs(v), minlength=n) + 1.0
    M = sp.csc_matrix((np.concatenate([v, dom.astype(v.dtype)]),
                       (np.concatenate([rows, np.arange(n)]), np.concatenate([cols, np.arange(n)]))), shape=(n, n))
    A = CSC.from_scipy(M)
    PW = pattern_from_matrix(sp.identity(n, format="csc"))
    F = D.factor(D.DeviceCSC.from_host(A), D.DeviceCSC.from_host(PW), D.RULE_FIXED,
                 Vfixed=D.DeviceCSC.from_host(A.pattern()), alg="S", prec="fp64")
    V = sp.csc_matrix((F.V.vals.cpu().numpy(), F.V.rowidx.cpu().numpy(), F.V.colptr.cpu().numpy()), shape=(n, n))
    W = F.W.vals.cpu().numpy()
    for seed in (1, 2):  # the first apply and a later one
        x = np.random.default_rng(seed).standard_normal(n).astype(A.vals.dtype)
        y = F.apply(torch.from_numpy(x).cuda()).cpu().numpy()
        ref = W * spl.spsolve_triangular(V.tocsr(), x, lower=lower)
        assert np.linalg.norm(y - ref, 1) <= 1e-11 * np.linalg.norm(ref, 1)
