"""The register-tile pass of small grids (the default blocking): the bits of one-step launches, at
region edges, remainders and grids smaller than a region's halo, for step counts that give one
short pass, equal passes and passes of two depths."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

RATES = (0.5, 0.2, 0.11, 0.1)
D = (0.05, 0.04, 0.01, 0.05, 0.0)
SIZES = [(1, 1), (2, 7), (5, 1), (31, 64), (36, 5), (64, 33), (65, 130), (130, 67), (257, 300)]


def _solver(nx, ny, lattice, precision, bc):
    s = L.Solver(nx, ny, RATES, d=D, bc=bc, precision=precision, lattice=lattice)
    if lattice == L.LATTICE_D2Q5_VARD:
        s.set_diffusivity_scale(*inputs.mobility_fields(nx, ny, seed=3, kind="random"))
    s.write(inputs.epidemic_state(nx, ny, seed=nx + 7 * ny))
    return s


@pytest.mark.parametrize("bc", [L.BC_PERIODIC, L.BC_NOFLUX])
@pytest.mark.parametrize("lattice,precision", [(L.LATTICE_D2Q5, L.FP32), (L.LATTICE_D2Q5, L.FP32_DEV),
                                               (L.LATTICE_D2Q9, L.FP32), (L.LATTICE_D2Q5_VARD, L.FP32)])
def test_tile_passes_give_the_bits_of_one_step_launches(lattice, precision, bc):
    for nx, ny in SIZES:
        for n in (2, 13, 29):
            ref = _solver(nx, ny, lattice, precision, bc)
            ref.set_blocking(1)
            ref.step(n)
            s = _solver(nx, ny, lattice, precision, bc)
            s.step(n)
            assert s.steps_done() == n
            a, b = s.read(dtype=np.float32), ref.read(dtype=np.float32)
            s.close()
            ref.close()
            assert np.array_equal(a.view(np.uint32), b.view(np.uint32)), (nx, ny, n)


def test_tile_passes_replay_from_a_captured_graph():
    """Steps enqueued under stream capture: the replayed graph advances the state as the calls did."""
    import torch
    ref = _solver(130, 67, L.LATTICE_D2Q5, L.FP32, L.BC_NOFLUX)
    ref.step(56)
    st = torch.cuda.Stream()
    s = L.Solver(130, 67, RATES, d=D, bc=L.BC_NOFLUX, precision=L.FP32, stream=st)
    s.write(inputs.epidemic_state(130, 67, seed=130 + 7 * 67))
    graph = torch.cuda.CUDAGraph()
    st.synchronize()
    with torch.cuda.graph(graph, stream=st):
        s.step(28)  # an even number of passes: the state is back in the buffer it started from
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    a, b = s.read(dtype=np.float32), ref.read(dtype=np.float32)
    assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
    s.close()
    ref.close()
