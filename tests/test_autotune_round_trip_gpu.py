"""sslbm_autotune returns one configuration and its time: on a grid small enough for the register tiles,
set_blocking(depth, seg_rows) on another handle steps in about the time reported, and both handles,
one on the tiles, one on that configuration, give the same bits."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

RATES = (0.5, 0.2, 0.11, 0.1)
D = (0.05, 0.04, 0.01, 0.05, 0.0)


def _ms_per_step(s, n=400):
    import torch
    s.step(n)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = 1e9
    for _ in range(5):
        a.record()
        s.step(n)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / n)
    return best


@pytest.mark.parametrize("nx,ny", [(128, 128), (300, 200)])
def test_autotuned_configuration_is_the_one_reported(nx, ny):
    st = inputs.epidemic_state(nx, ny, seed=nx)
    tuned = L.Solver(nx, ny, RATES, d=D, bc=L.BC_NOFLUX, precision=L.FP32)
    tuned.write(st)
    depth, seg, ms = tuned.autotune(60.0)
    assert tuned.get_blocking() == (depth, seg)
    other = L.Solver(nx, ny, RATES, d=D, bc=L.BC_NOFLUX, precision=L.FP32)
    other.set_blocking(depth, seg)
    other.write(st)
    # the two are separate timings of the same passes; the tiles take less than a third of either
    assert _ms_per_step(other) < 2.0 * ms
    assert _ms_per_step(other) > 0.4 * ms
    for s in (tuned, other):
        s.write(st)
        s.step(50)
    np.testing.assert_array_equal(tuned.read(), other.read())
    tuned.close()
    other.close()
