"""What the first apply leaves allocated: W by rows in V's order, V in the one
form that its solves use, the right-hand side's buffer -- and none of the
preparation's scratch, whose memory is another set-up's as soon as the call has
enqueued its work.  The sizes below are those arrays' own, each rounded up to the
allocator's 256 bytes."""
import pytest
import scipy.sparse as sp

import oracle as O
from tests.test_gpu_parity import run_gpu
from workloads import CSC, diagonal_pattern, make_workload, pattern_of

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import build, diaf
    build.build()
    return diaf


# bytes per row of V's form
PACKED_REAL = 4 * 4 + 4 * 8 + 8 * 4 + 6 * 8  # four entries, eight slot words and six merged values
PACKED_CPLX = 4 * 4 + 4 * 16


@pytest.mark.parametrize("name,form", [("convdiff48_A2", PACKED_REAL), ("helmholtz40", PACKED_CPLX),
                                       ("real_band", None), ("complex_band", None)])
def test_held_after_first_apply(D, name, form):
    """The bands are upper triangular with six entries beside the diagonal, beyond the packed form (W diagonal, V on
    the band)."""
    if form:
        w = make_workload(name)
        A, PW, rule, how = w.A, w.PW, (w.vrule, w.budget), dict(alg="S", prec="mixed32", tie_tol=w.tie_tol)
    else:
        c = 1j if name == "complex_band" else 1.0
        A = CSC.from_scipy(sp.diags([8.0] + 6 * [c], range(7), shape=(2000, 2000)).tocsc())
        PW, rule, how = diagonal_pattern(A.n), (O.RULE_FIXED, None, pattern_of(A)), dict(alg="S", prec="mixed32")
    F = run_gpu(D, A, PW, *rule, **how)
    longest = int(torch.bincount(F.V.rowidx.long(), minlength=A.n).max()) - 1
    assert (longest <= 4) == (form is not None)
    before = D.device_memory_in_use()
    x = torch.ones(A.n, dtype=F.V.vals.dtype, device="cuda")
    y = F.apply(x).clone()
    torch.cuda.synchronize()
    held = D.device_memory_in_use() - before
    v = F.V.vals.element_size()
    n, nnzw, nnzv = A.n, F.W.rowidx.numel(), F.V.rowidx.numel()
    rows = 4 * (n + 1) + nnzw * (4 + v)                # W
    rows += 4 * (n + 1) + n * (v + 4 + v)              # level pointers, 1 / diag, row map, t
    rows += n * form if form else 4 * (n + 1) + (nnzv - n) * (4 + v)
    assert held <= rows + 16 * 256, (held, rows)
    # the memory given back is used by other set-ups now; the solves do not miss it
    others = [run_gpu(D, A, PW, *rule, **how) for _ in range(3)]
    for G in others:
        G.apply(2 * x)
    assert torch.equal(F.apply(x), y)
    for G in others + [F]:
        G.close()
    assert D.device_memory_in_use() <= before
