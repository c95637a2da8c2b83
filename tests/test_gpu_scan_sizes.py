"""The prefix sums behind the column pointers (gathered entries, V's counts,
rows of W) at the sizes where their launch form changes -- one block, blocks
that add up the totals before them, totals scanned on their own -- and one
element to either side: V's column pointers against the budgets' running sum,
and the apply against V times its result (relative residual within 1e-12: one
entry of W per column, diagonally dominant columns)."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
from tests._parity import host_factors
from workloads import CSC

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 3 * 1024, 2048 * 1024, 2048 * 1024 + 1])
def test_scan_edges(n):
    from paper_1208_3573_gb300 import diaf
    rng = np.random.default_rng(n)
    A = sp.diags([rng.uniform(4.0, 8.0, n)] + [rng.uniform(-1.0, 1.0, n - d) for d in (1, 2, 3) if d < n],
                 [0] + [d for d in (1, 2, 3) if d < n]).tocsc()
    A.sort_indices()
    PW = CSC.from_scipy(sp.identity(n, format="csc"))
    budget = np.where(np.arange(n) % 3 == 1, 2, 1).astype(np.int32)
    hA = CSC.from_scipy(A)
    dA, dP = diaf.DeviceCSC.from_host(hA), diaf.DeviceCSC.from_host(PW)
    F = diaf.factor(dA, dP, O.RULE_UPPER, torch.from_numpy(budget).cuda(), alg="S", prec="fp64")
    x = rng.standard_normal(n)
    y = F.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    F.sync()
    f = host_factors(F)
    cp = np.concatenate([[0], np.cumsum(O.vcount(hA, PW, O.RULE_UPPER, budget))])
    assert np.array_equal(f["Vcp"], cp)
    V = sp.csc_matrix((f["Vv"], f["Vri"], f["Vcp"]), (n, n))
    assert np.linalg.norm(V @ (y / f["Wv"]) - x) <= 1e-12 * np.linalg.norm(x)
    F.close()
