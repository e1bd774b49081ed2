"""The FP64 one-step kernel at the edges of its work split (equal shares per SM up to 1024 cells
each, 64-cell blocks beyond) against the FP64 oracle: three steps of at most 40 rounded operations on
a cell, so 3 * 40 * 2^-53 = 1.3e-14 of the compartment's largest value, doubled for the oracle's own."""
import numpy as np
import pytest

import oracle
from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

D = (0.05, 0.04, 0.01, 0.05, 0.0)
RATES = (0.5, 0.2, 0.11, 0.1)


@pytest.mark.parametrize("bc", [L.BC_PERIODIC, L.BC_NOFLUX])
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 1), (151, 1), (1, 153), (13, 11), (200, 200), (395, 394), (397, 393),
                                   (64, 2433), (1023, 153)])
def test_equal_shares_match_the_oracle(nx, ny, bc):
    st = inputs.epidemic_state(nx, ny, seed=nx + ny)
    s = L.Solver(nx, ny, RATES, d=D, bc=bc, precision=L.FP64)
    s.write(st)
    s.step(3)
    got = s.read()
    s.close()
    want = oracle.sslbm_run(st, [oracle.tau_from_d(v) for v in D[:4]], RATES, 1.0, bc, 3)
    err = np.abs(got - want).reshape(5, -1).max(axis=1) / np.abs(want).reshape(5, -1).max(axis=1)
    assert err.max() <= 2.6e-14, err
