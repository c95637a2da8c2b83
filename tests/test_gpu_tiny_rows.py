"""Rows of A far below the others (1e-50, below every FP32 number beside them):
an entry that is zero in FP32 still belongs to the FP64 products, so v = T(I_j,:) w
holds row by row to the rounding of a k-term sum (v_jj of such a row is zero only where w
is zero on all of the row's columns), and the factors can be applied."""
import numpy as np
import pytest

from tests._parity import host_factors
from workloads import CSC, make_workload

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import build, diaf
    build.build()
    return diaf


@pytest.mark.parametrize("alg", ["S", "Q"])
@pytest.mark.parametrize("name,small", [("convdiff48_A2", 1), ("convdiff48_A2", 2), ("helmholtz40", 1),
                                        ("lognormal16", 1), ("powerlaw6k", 1)])
def test_rows_of_v(D, name, small, alg):
    w = make_workload(name)
    rng = np.random.default_rng(11)
    scale = np.ones(w.n)
    scale[rng.choice(w.n, w.n // 20, replace=False)] = 1e-50
    A = CSC(w.n, w.A.colptr, w.A.rowidx, w.A.vals * scale[w.A.rowidx])
    F = D.factor(D.DeviceCSC.from_host(A), D.DeviceCSC.from_host(w.PW), w.vrule, torch.from_numpy(w.budget).cuda(),
                 alg=alg, prec="mixed32", tie_tol=w.tie_tol, tuning={"small_tiles": small})
    g = host_factors(F)
    M = A.to_scipy().tocsr()
    absM = abs(M)
    bad = []
    for j in range(w.n):
        J, wj = g["Wri"][g["Wcp"][j]:g["Wcp"][j + 1]], g["Wv"][g["Wcp"][j]:g["Wcp"][j + 1]]
        I, vj = g["Vri"][g["Vcp"][j]:g["Vcp"][j + 1]], g["Vv"][g["Vcp"][j]:g["Vcp"][j + 1]]
        if alg == "S":
            exact = M[I][:, J] @ wj
            bound = 8 * (J.size + 8) * EPS * (absM[I][:, J] @ np.abs(wj))
            if (np.abs(vj - exact) > bound).any():
                bad.append(j)
    assert not bad, (len(bad), bad[:5])
    if alg == "S" and name == "helmholtz40":  # every v_jj is above its rounding here
        diag = F.V.vals[F.V.rowidx == torch.repeat_interleave(torch.arange(w.n, device="cuda"), F.V.colptr.diff())]
        assert (diag != 0).all()
        F.apply(torch.ones(w.n, dtype=F.V.vals.dtype, device="cuda"))
        torch.cuda.synchronize()
