"""The streaming one-step kernel on the edges of its strips (64 columns, whole 16-byte groups and
single columns copied apart) and of its row segments (one row each on small grids), every
update, against the FP64 oracle: one step, relative max-norm per compartment.  A cell's update
is at most 30 rounded operations on values of its own size, so FP32 stays within 30 u = 1.8e-6
and the double word within 30 * 10 u^2 = 1.1e-12 of the compartment's largest value."""
import numpy as np
import pytest

import oracle
from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

D = (0.05, 0.04, 0.01, 0.05, 0.0)
RATES = (0.5, 0.2, 0.11, 0.1)


@pytest.mark.parametrize("bc", [L.BC_PERIODIC, L.BC_NOFLUX])
@pytest.mark.parametrize("nx,ny", [(1, 3), (3, 1), (5, 7), (62, 9), (63, 5), (64, 33), (65, 2), (66, 130), (127, 1),
                                   (130, 257), (195, 64)])
def test_one_step_matches_the_oracle_at_strip_and_segment_edges(nx, ny, bc):
    st = inputs.epidemic_state(nx, ny, seed=nx * 1000 + ny)
    tau = [oracle.tau_from_d(v) for v in D[:4]]
    kx, ky = inputs.mobility_fields(nx, ny, seed=5, kind="random")
    cases = [(L.LATTICE_D2Q5, p, tol) for p, tol in ((L.FP32, 1.8e-6), (L.FP32_DEV, 1.8e-6), (L.FP32_SPLIT, 1.8e-6),
                                                     (L.FP32_KAHAN, 1.8e-6), (L.FP64_DW, 1.1e-12))]
    cases += [(L.LATTICE_D2Q9, L.FP32, 1.8e-6), (L.LATTICE_D2Q5_VARD, L.FP32, 1.8e-6)]
    for lattice, precision, tol in cases:
        s = L.Solver(nx, ny, RATES, d=D, bc=bc, precision=precision, lattice=lattice)
        if lattice == L.LATTICE_D2Q5_VARD:
            s.set_diffusivity_scale(kx, ky)
            want = oracle.sslbm_vard_run(st, tau, RATES, kx, ky, 1.0, bc, 1)
        else:
            run = oracle.sslbm9_run if lattice == L.LATTICE_D2Q9 else oracle.sslbm_run
            want = run(st, tau, RATES, 1.0, bc, 1)
        s.write(st)
        s.step(1)
        got = s.read()
        s.close()
        err = np.abs(got - want).reshape(5, -1).max(axis=1) / np.abs(want).reshape(5, -1).max(axis=1)
        assert err.max() <= tol, (lattice, precision, err)
