"""Where the finite-difference reference keeps its state: the first five contiguous planes [5][ny][nx] of
the workspace after any number of steps, so that a captured call can be replayed for odd and even n,
also with other calls between the replays."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import sslbm as L

from test_fd4_gpu import D, RATES, _state

pytestmark = pytest.mark.gpu


def _solver(nx, ny, bc, precision, order=4):
    f = L.Fd4(nx, ny, RATES, D, dx=0.5, dt=0.8, bc=bc, precision=precision, order=order)
    st = _state(nx, ny, nx + ny)
    f.write(st.astype(np.float32) if precision == L.FP32 else st)
    return f


def _bits(a):
    return np.ascontiguousarray(a).view(np.uint8)


@pytest.mark.parametrize("precision,dtype", [(L.FP32, np.float32), (L.FP64, np.float64)])
@pytest.mark.parametrize("nx,ny,bc", [(131, 33, L.BC_NOFLUX), (128, 40, L.BC_PERIODIC), (5, 70, L.BC_PERIODIC)])
def test_state_is_the_workspace_s_first_planes(nx, ny, bc, precision, dtype):
    f = _solver(nx, ny, bc, precision)
    for n in (1, 1, 2, 3):
        f.step(n)
        got = f.read(dtype=dtype)
        raw = f.ws[:got.nbytes].cpu().numpy()
        assert np.array_equal(raw, _bits(got).reshape(-1)), n


@pytest.mark.parametrize("n", [1, 2, 3])
@pytest.mark.parametrize("precision,dtype", [(L.FP32, np.float32), (L.FP64, np.float64)])
def test_captured_steps_replay_for_odd_and_even_counts(n, precision, dtype):
    import torch
    nx, ny = 133, 41
    a, b = _solver(nx, ny, L.BC_NOFLUX, precision), _solver(nx, ny, L.BC_NOFLUX, precision)
    stream = torch.cuda.Stream()
    f = L.Fd4(nx, ny, RATES, D, dx=0.5, dt=0.8, bc=L.BC_NOFLUX, precision=precision, stream=stream)
    f.step(1)  # the kernels' attributes are set before the capture
    f.write(a.read(dtype=dtype))
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        f.step(n)
    torch.cuda.synchronize()
    total = 0
    for eager in (0, 1, 0):  # steps outside the graph between the replays
        with torch.cuda.stream(stream):
            graph.replay()
        f.step(eager)
        total += n + eager
        b.step(n + eager)
        stream.synchronize()
        assert np.array_equal(_bits(f.read(dtype=dtype)), _bits(b.read(dtype=dtype))), total
    for s in (a, b, f):
        s.close()
