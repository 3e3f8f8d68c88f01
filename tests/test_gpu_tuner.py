"""Tile choice of float64 handles: fixed only on the grids where it was found to be the fastest."""
import pytest

from paper_2412_17445_gb300 import binding as B
from paper_2412_17445_gb300 import microstructure as ms

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2412_17445_gb300 import build
    build.build()
    B.lib()


@pytest.mark.parametrize("shape,timed", [((36, 96), False), ((54, 432), False), ((54, 486), True), ((12, 1458), True),
                                         ((324, 972), True), ((648, 24), True)])
def test_float64_tiles_timed_off_the_measured_range(shape, timed):
    """One candidate is four applies of three kernels; long rows and more than 608 rows are timed with
    two candidates at least (rows of 972 points leave one row pair a block, with 1, 2 or 4 columns)."""
    inp = ms.random_rve(shape, 3, notch=False)
    eps, E, phi, H = ms.random_state(inp, 4)
    g = B.RVE(inp)
    g.set_state(B.mandel_from_tensor(eps), phi, H, E)
    g.linearize(B.RVE_CTRL_CRACK, 1.0)
    before = g.kernel_launches()
    g.autotune()
    n = g.kernel_launches() - before
    assert n >= 24 if timed else n == 12
    g.close()
