"""The diagnostics reduction at the widths where its rows per block change, alone and in an ensemble: the
same bits both ways, and the exact sums to rounding."""
import math

import numpy as np
import pytest

from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

RATES = (0.5, 0.2, 0.11, 0.1)
D = (0.05, 0.04, 0.01, 0.05, 0.0)
SIZES = [(4, 1), (64, 5), (2044, 7), (2048, 9), (4092, 3), (4096, 5), (4, 5000), (12000, 30)]


@pytest.mark.parametrize("precision", [L.FP32, L.FP32_DEV, L.FP32_SPLIT])
def test_grid_and_ensemble_totals_agree(precision):
    ens = L.Ensemble([dict(nx=nx, ny=ny, rates=RATES, d=D, s_ref=1.0) for nx, ny in SIZES], precision=precision)
    for i, (nx, ny) in enumerate(SIZES):
        ens.write(i, np.random.default_rng(i).uniform(0, 1, (5, ny, nx)))
    for _ in range(2):
        totals, peak = ens.diagnostics()
        for i, (nx, ny) in enumerate(SIZES):
            st = ens.read(i)
            want = [math.fsum(st[c].ravel()) for c in range(5)]
            np.testing.assert_allclose(totals[i], want, rtol=1e-12)
            assert peak[i] == st[2].max()
            s = L.Solver(nx, ny, RATES, d=D, precision=precision, s_ref=1.0)
            s.write(np.random.default_rng(i).uniform(0, 1, (5, ny, nx)))
            if s.steps_done() == ens_steps(ens):
                t, p = s.diagnostics()
                assert np.array_equal(t, totals[i]) and p == peak[i]
            s.close()
        ens.run(4)  # the reduction's scratch lies in the spare buffer, which the run overwrites
    ens.close()


def ens_steps(ens):
    return L.sslbm_ensemble_steps_done(ens.e)
