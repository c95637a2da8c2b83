"""bench.py's flop count charges a Jacobi SVD to the columns whose kernel runs
one, tile by tile, whatever bucket took the most time."""
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

M = np.array([20, 32, 33, 64, 65, 70, 600])
K = np.array([10, 16, 16, 32, 20, 33, 60])


def test_columns_by_tile():
    large = [False, False, False, False, True, True, True]
    for prec, cplx in (("mixed32", False), ("mixed32", True), ("fp64", False)):
        assert bench.svd_columns(M, K, "S", prec, cplx).tolist() == large
    assert bench.svd_columns(M, K, "S", "fp64", True).all()
    assert bench.svd_columns(M, K, "Q", "mixed32", False).all()


def test_flops_are_the_sum_over_columns():
    L = np.full(M.size, 5)
    svd = bench.svd_columns(M, K, "S", "mixed32", False)
    each = [bench.algorithmic_flops(M[i:i + 1], K[i:i + 1], L[i:i + 1], "S", False, svd=bool(svd[i]))
            for i in range(M.size)]
    got = bench.algorithmic_flops(M, K, L, "S", False, svd=svd)
    assert np.allclose(got, np.sum(each, axis=0), rtol=1e-12)
    assert not np.isclose(got[0], bench.algorithmic_flops(M, K, L, "S", False, svd=False)[0], rtol=1e-3)
