"""The launches an FP32 step of the finite-difference reference is made of -- pairs of stages on tiles of 8
or 16 rows, the four stage launches of narrow and of small no-flux grids, an odd last step in place or by
a pair and a copy -- on grids that take each: bitwise against the float32 evaluation."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import sslbm as L

from test_fd4_gpu import D, RATES, _fd4_float32, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [4, 2])
@pytest.mark.parametrize("bc", [L.BC_PERIODIC, L.BC_NOFLUX])
@pytest.mark.parametrize("nx,ny", [(3, 9000), (33, 1500), (64, 900), (5000, 8), (129, 3000), (800, 600), (801, 600),
                                   (640, 512), (1536, 1400)])
def test_every_route_is_the_float32_evaluation(nx, ny, bc, order):
    st = _state(nx, ny, nx + 3 * ny).astype(np.float32)
    f = L.Fd4(nx, ny, RATES, D, dx=0.5, dt=0.8, bc=bc, precision=L.FP32, order=order)
    f.write(st)
    ref = st
    for steps in (1, 2, 3):
        f.step(steps)
        ref = _fd4_float32(ref, D, RATES, 0.5, 0.8, bc, steps, order)
        got = f.read(dtype=np.float32)
        assert np.array_equal(got.view(np.uint32), ref.view(np.uint32)), steps
    f.close()
