"""The blocked D2Q9 kernel with walls where the last strip is narrower than the depth: the wall's column then
lies within the steps' reach of the strip before it.  Every width from one column beyond a strip's edge to
past the depth, the bits of one step per launch."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

RATES = (0.5, 0.2, 0.11, 0.1)
D = (0.05, 0.04, 0.01, 0.05, 0.0)


@pytest.mark.parametrize("strips", [1, 2])
@pytest.mark.parametrize("depth", [2, 3, 4, 5, 6, 7, 8])
def test_last_strip_narrower_than_the_depth(depth, strips):
    cols = 128 - 8 * ((depth + 3) // 4)
    for nx in range(strips * cols + 1, strips * cols + depth + 3):
        ny = 21
        st = inputs.epidemic_state(nx, ny, seed=nx)
        s = L.Solver(nx, ny, RATES, d=D, bc=L.BC_NOFLUX, precision=L.FP32, lattice=L.LATTICE_D2Q9)
        s.set_blocking(1, 0)
        s.write(st)
        s.step(2 * depth)
        want = s.read()
        s.set_blocking(depth, 0)
        s.write(st)
        s.step(2 * depth)
        np.testing.assert_array_equal(s.read(), want, err_msg=str(nx))
        s.close()
