"""Several BGK steps per pass (FP32): the populations of one-step launches, bit for bit, at region
edges, remainders, walls and grids smaller than a region's halo, for step counts that give one
pass, equal passes and passes of two depths."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

RATES = (0.5, 0.2, 0.11, 0.1)
D = (0.05, 0.04, 0.01, 0.05, 0.0)


@pytest.mark.parametrize("bc", [L.BC_PERIODIC, L.BC_NOFLUX])
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (5, 1), (1, 9), (17, 9), (56, 8), (57, 25), (64, 33), (130, 67),
                                   (900, 161), (903, 700)])
def test_passes_give_the_populations_of_one_step_launches(nx, ny, bc):
    st = inputs.epidemic_state(nx, ny, seed=nx + 5 * ny)
    for n in (2, 4, 9):
        one, many = (L.Solver(nx, ny, RATES, d=D, bc=bc, precision=L.FP32, schemes=L.WANT_BGK) for _ in range(2))
        for s in (one, many):
            s.write(st, scheme=L.SCHEME_BGK)
        for _ in range(n):
            one.bgk_step(1)
        many.bgk_step(n)
        assert many.steps_done(L.SCHEME_BGK) == n
        assert np.array_equal(one.checkpoint(), many.checkpoint()), n
        one.close()
        many.close()
