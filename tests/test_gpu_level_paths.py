"""The level solve of a packed real V: that each rule leads to the form it
should (apply_form), on the paths that the other suite's sizes do not reach --
groups whose entries lie beyond the window, merged rows that do not fit among
more levels than shared memory has pointers for -- and what grouping does to the
result where V's rows are not dominated by their diagonals.

W is diagonal and V's pattern is A's, so V is A up to column signs and y solves
A y = x.  The reference is the row by row substitution in extended precision;
the bound is sixteen times the error of the same substitution in FP64 (the
grouped solve has the same error bound, |V^-1| |V| |t| eps, with up to four
levels' products formed beforehand; measured on 21 random problems with multipliers
of 0.3 to 100: at most 2.1 times)."""
import numpy as np
import pytest
import scipy.sparse as sp

from tests._problems import pattern_from_matrix
from tests.test_gpu_level_groups import layered
from workloads import CSC

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FULL, FAR = 1, 2


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import build, diaf
    build.build()
    return diaf


def factored(D, M):
    A = CSC.from_scipy(sp.csc_matrix(M))
    PW = pattern_from_matrix(sp.identity(A.n, format="csc"))
    return D.factor(D.DeviceCSC.from_host(A), D.DeviceCSC.from_host(PW), D.RULE_FIXED,
                    Vfixed=D.DeviceCSC.from_host(A.pattern()), alg="S", prec="fp64")


def substitution(M, x, dtype):
    """A y = x for an upper triangular A, row by row from the last."""
    R = M.tocsr()
    R.sort_indices()
    n = R.shape[0]
    y = np.zeros(n, dtype)
    ptr, idx, val = R.indptr, R.indices, R.data.astype(dtype)
    for i in range(n - 1, -1, -1):
        a, b = ptr[i], ptr[i + 1]
        s = x[i].astype(dtype)
        for q in range(a + 1, b):
            s = s - val[q] * y[idx[q]]
        y[i] = s / val[a]
    return y


def neighbours(widths):
    """Rows that depend on the two next to them in the level before, as a stencil's: five merged entries at most."""
    width, n = widths[0], sum(widths)
    i = np.arange(n - width)
    return n, np.repeat(i, 2), np.stack([i + width, i - i % width + width + (i + 1) % width], 1).ravel()


CASES = {  # level widths, entries per row (None: neighbours), far, levels per group, flags
    "grouped": ([256] * 41, None, False, 4, 0),
    "grouped_full": ([256] * 10, 2, False, 4, FULL),
    "grouped_far": ([256] * 80, 2, True, 4, FAR),
    "full_pointers_beyond_smem": ([4] * 9000, 4, False, 4, FULL),
    "wide": ([1500] * 4, 2, False, 1, 0),
    "rows": ([50] * 12, 5, True, 0, 0),
}


@pytest.mark.parametrize("case,mult", [(c, m) for c in CASES for m in (0.25, 4.0)
                                       if m < 1.0 or len(CASES[c][0]) < 500])  # y grows by the level
def test_form_and_error(D, case, mult):
    """mult: multipliers v_ij / v_ii of half to all of it; the error is taken level by level."""
    widths, parents, far, group, flags = CASES[case]
    n, rows, cols = layered(widths, parents, 5, far) if parents else neighbours(widths)
    rng = np.random.default_rng(9)
    v = mult * rng.uniform(0.5, 1.0, rows.size) * rng.choice([-1.0, 1.0], rows.size)
    M = sp.csc_matrix((np.concatenate([v, np.ones(n)]), (np.concatenate([rows, np.arange(n)]),
                                                         np.concatenate([cols, np.arange(n)]))), shape=(n, n))
    F = factored(D, M)
    x = rng.standard_normal(n)
    y = F.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    got = F.apply_form()
    assert got[0] == group and (got[1] & flags) == flags and (flags or got[1] == 0), got
    ref, seq = substitution(M, x, np.longdouble), substitution(M, x, np.float64)
    ends = n - np.cumsum([0] + list(widths))

    def err(t):
        return max(float(np.linalg.norm((t[b:a] - ref[b:a]) / np.max(np.abs(ref[b:a])))
                         / np.linalg.norm(ref[b:a] / np.max(np.abs(ref[b:a])))) for a, b in zip(ends, ends[1:]))
    assert err(y) <= 16.0 * max(err(seq), np.finfo(np.float64).eps), (err(y), err(seq))


def test_products_out_of_range(D):
    """Multipliers whose products overflow: the zeros of a sparse right-hand side stay zeros."""
    n = 40
    M = sp.diags([np.ones(n), np.full(n - 1, 1e200)], [0, 1]).tocsc()
    F = factored(D, M)
    x = np.zeros(n)
    x[0] = 3.0  # the row that is solved last
    y = F.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    assert np.array_equal(np.abs(y), x)
    assert F.apply_form() == (4, FULL)
