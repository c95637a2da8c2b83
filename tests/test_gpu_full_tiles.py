"""Full tiles of 17 to 32 columns: every lane of the Gram matrix has m k
entries to go over (10 m k >= m (k + 20)), so the wide DIAF-S warp kernels form
it densely, which banded tiles of that width never do.  Every value type and
precision against the oracle, with the tolerances of the parity suites."""
import pytest

from tests.test_gpu_smallest import banded, check, window

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    from paper_1208_3573_gb300 import build, diaf
    build.build()
    return diaf


@pytest.mark.parametrize("prec", ["fp64", "mixed32"])
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,k", [(60, 17), (64, 25), (63, 32)])
def test_full_tiles(D, n, k, cplx, prec):
    check(D, banded(n, n + k, cplx, bands=n - 1), window(n, k), prec)
