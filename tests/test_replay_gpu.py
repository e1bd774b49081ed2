"""Captured step calls replay: where the default blocking takes passes of its own depths (register tiles,
deeper pipeline passes, multi-step BGK passes) a captured call of n >= 2 steps leaves the state in the
buffer it started from, and calls between the replays keep the parity of the plain cut."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

RATES = (0.5, 0.2, 0.11, 0.1)
D = (0.05, 0.04, 0.01, 0.05, 0.0)


def _solver(nx, ny, lattice, precision, schemes, stream=None):
    s = L.Solver(nx, ny, RATES, d=D, bc=L.BC_NOFLUX, precision=precision, lattice=lattice, schemes=schemes, stream=stream)
    if lattice == L.LATTICE_D2Q5_VARD:
        s.set_diffusivity_scale(*inputs.mobility_fields(nx, ny, seed=3, kind="random"))
    return s


# between: an even number of passes of the plain cut (depth 4; BGK one step each)
@pytest.mark.parametrize("nx,ny,lattice,precision,bgk,between", [
    (130, 67, L.LATTICE_D2Q5, L.FP32, False, 8), (513, 300, L.LATTICE_D2Q5, L.FP32_DEV, False, 5),
    (96, 90, L.LATTICE_D2Q9, L.FP32, False, 8), (300, 200, L.LATTICE_D2Q5_VARD, L.FP32, False, 16),
    (1024, 900, L.LATTICE_D2Q5, L.FP32_SPLIT, False, 8), (1024, 900, L.LATTICE_D2Q5, L.FP32_KAHAN, False, 13),
    (2100, 1800, L.LATTICE_D2Q5_VARD, L.FP32, False, 8), (70, 50, L.LATTICE_D2Q5, L.FP32, True, 4)])
def test_captured_calls_replay(nx, ny, lattice, precision, bgk, between):
    import torch
    scheme = L.SCHEME_BGK if bgk else L.SCHEME_SSLBM
    schemes = L.WANT_BGK if bgk else L.WANT_SSLBM
    st = inputs.epidemic_state(nx, ny, seed=nx + ny)
    ref = _solver(nx, ny, lattice, precision, schemes)
    stream = torch.cuda.Stream()
    s = _solver(nx, ny, lattice, precision, schemes, stream)
    step, ref_step = (s.bgk_step, ref.bgk_step) if bgk else (s.step, ref.step)
    step(8)  # kernel attributes are set before the capture
    for n in (2, 3, 4, 6, 11, 20):
        s.write(st, scheme=scheme)
        ref.write(st, scheme=scheme)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            step(n)
        torch.cuda.synchronize()
        for eager in (0, 0, between, 0):
            with torch.cuda.stream(stream):
                graph.replay()
            step(eager)
            ref_step(n)
            ref_step(eager)
        stream.synchronize()
        np.testing.assert_array_equal(s.read(scheme=scheme), ref.read(scheme=scheme), err_msg=str(n))
    s.close()
    ref.close()
