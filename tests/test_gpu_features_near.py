"""Feature f4, log |a_cc| / |a_jj|, of nearly equal diagonals: correct to the
rounding of FP32 (the bound is two of its rounding units) however small it is and
whatever the diagonals' size."""
import numpy as np
import pytest
import scipy.sparse as sp

from workloads import CSC, patterns as pats

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import build, diaf
    build.build()
    return diaf


# (a complex modulus is the root of a sum of squares, so its sizes end at 1e+-150)
@pytest.mark.parametrize("size,cplx", [(1.0, False), (4e7, False), (1e250, False), (3e-200, False),
                                       (1.0, True), (4e7, True), (1e120, True), (3e-100, True)])
def test_log_ratio(D, size, cplx):
    n = 64
    rng = np.random.default_rng(2)
    d = size * (1.0 + np.where(np.arange(n) % 5 == 0, 0.0, rng.choice([-1.0, 1.0], n)
                               * 10.0 ** rng.uniform(-15.5, 0.3, n)).clip(-0.9))
    M = sp.diags([d, np.full(n - 1, 0.3 * size), np.full(n - 1, 0.2 * size)], [0, 1, -1]).tocsc()
    A = CSC.from_scipy(M.astype(np.complex128) if cplx else M)
    P = pats.pattern_of(A)
    f = D.propose_features(D.DeviceCSC.from_host(A), D.DeviceCSC.from_host(P)).cpu().numpy()[:, 4]
    col = np.repeat(np.arange(n), np.diff(P.colptr))
    a, b = d[P.rowidx], d[col]
    near = np.abs(a - b) < 0.5 * np.minimum(a, b)
    e = np.where(near, np.log1p((a - b) / b), np.log(a / size) - np.log(b / size))
    np.testing.assert_allclose(f, e, rtol=2.4e-7, atol=0)
