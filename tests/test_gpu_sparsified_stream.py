"""sparsified_powers on a stream of the caller's own: the pattern is complete
when the call returns, whatever the one-pass (keep <= 64) or two-pass form
left to do last, and the work waits for what the current stream had enqueued
before the call."""
import numpy as np
import pytest

from oracle.sparsified import sparsified_powers as oracle_sp
from workloads import operators as ops

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SLEEP = 40_000_000  # clock cycles, about 20 ms


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import build, diaf
    build.build()
    return diaf


@pytest.mark.parametrize("keep", [0, 5, 64, 65])
def test_complete_on_return(D, monkeypatch, keep):
    A = ops.lognormal3d(8, seed=4)
    dA = D.DeviceCSC.from_host(A)
    side = torch.cuda.Stream()
    L = D.lib()

    def late(real):
        def f(*args):
            with torch.cuda.stream(side):
                torch.cuda._sleep(SLEEP)
            return real(*args)
        return f

    for name in ("diaf_sparsified_pack", "diaf_sparsified_fill"):  # the last step comes late
        monkeypatch.setattr(L, name, late(getattr(L, name)))
    torch.cuda.synchronize()
    P = D.sparsified_powers(dA, 2, 0, keep, stream=side)
    assert side.query()
    o = oracle_sp(A, 2, 0, keep)
    np.testing.assert_array_equal(P.colptr.cpu().numpy(), o.colptr)
    np.testing.assert_array_equal(P.rowidx.cpu().numpy(), o.rowidx)


@pytest.mark.parametrize("keep", [0, 5])
def test_waits_for_the_current_stream(D, keep):
    """The output arrays come from the current stream's memory, where enqueued
    work may still use them, and A may still be in the making there."""
    A = ops.lognormal3d(8, seed=4)
    ready = D.DeviceCSC.from_host(A)
    dA = D.DeviceCSC(A.n, ready.colptr, ready.rowidx, torch.ones_like(ready.vals))
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(SLEEP)
    dA.vals.copy_(ready.vals)
    P = D.sparsified_powers(dA, 2, 0, keep, stream=side)
    o = oracle_sp(A, 2, 0, keep)
    np.testing.assert_array_equal(P.colptr.cpu().numpy(), o.colptr)
    np.testing.assert_array_equal(P.rowidx.cpu().numpy(), o.rowidx)
