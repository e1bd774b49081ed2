"""The pipeline's 32-bit rows and columns (varying diffusion, Kahan, D2Q9) and the split storage at explicit
depths, on grids smaller than the halo, on strip edges (112 and 120 columns) and ragged ones, where the
default blocking would take register tiles or depth 4: the bits of one step per launch."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

D = (0.05, 0.04, 0.01, 0.05, 0.0)
RATES = (0.5, 0.2, 0.11, 0.1)


@pytest.mark.parametrize("lattice,precision", [(L.LATTICE_D2Q5, L.FP32_KAHAN), (L.LATTICE_D2Q5, L.FP32_SPLIT),
                                               (L.LATTICE_D2Q5_VARD, L.FP32), (L.LATTICE_D2Q9, L.FP32)])
@pytest.mark.parametrize("bc", [L.BC_PERIODIC, L.BC_NOFLUX])
@pytest.mark.parametrize("nx,ny", [(1, 2), (3, 5), (113, 40), (120, 33), (224, 9), (243, 131)])
def test_every_depth_gives_the_bits_of_single_steps(nx, ny, bc, lattice, precision):
    st = inputs.epidemic_state(nx, ny, seed=nx + ny)
    s = L.Solver(nx, ny, RATES, d=D, bc=bc, precision=precision, lattice=lattice)
    if lattice == L.LATTICE_D2Q5_VARD:
        s.set_diffusivity_scale(*inputs.mobility_fields(nx, ny, seed=5, kind="random"))
    s.set_blocking(1, 0)
    s.write(st)
    s.step(17)
    want = s.read()
    for k in (4, 6, 8):
        s.set_blocking(k, 0)
        s.write(st)
        s.step(17)
        np.testing.assert_array_equal(s.read(), want, err_msg=str(k))
    s.close()
