"""The FP32 two-stage launches of the finite-difference reference at the edges of their tiles (128
columns; 16 rows, or 8 below one wave of those): bitwise against the float32 evaluation, widths
with and without aligned groups of four, grids narrower than the stencil, odd and even step
counts (the state alternates between two buffers), and reads between steps."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import sslbm as L

from test_fd4_gpu import D, RATES, _fd4_float32, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [4, 2])
@pytest.mark.parametrize("bc", [L.BC_PERIODIC, L.BC_NOFLUX])
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 1), (1, 40), (127, 17), (128, 16), (129, 15), (130, 34), (256, 8),
                                   (1030, 770), (1024, 609)])
def test_pairs_of_stages_are_the_float32_evaluation(nx, ny, bc, order):
    st = _state(nx, ny, nx + 3 * ny)
    f = L.Fd4(nx, ny, RATES, D, dx=0.5, dt=0.8, bc=bc, precision=L.FP32, order=order)
    f.write(st.astype(np.float32))
    ref = st.astype(np.float32)
    for steps in (1, 2):
        f.step(steps)
        ref = _fd4_float32(ref, D, RATES, 0.5, 0.8, bc, steps, order)
        f.read()  # FP64 conversion through the scratch buffers leaves the state alone
        got = f.read(dtype=np.float32)
        assert np.array_equal(got.view(np.uint32), ref.view(np.uint32)), steps
    f.close()
