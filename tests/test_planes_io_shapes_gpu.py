"""Device transfers on grids that take each launch shape of the transfer kernel -- narrow and tall, ragged and
aligned, small CTAs and four rows per thread: the same values as the host transfers."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

RATES = (0.5, 0.2, 0.11, 0.1)
D = (0.05, 0.04, 0.01, 0.05, 0.0)


@pytest.mark.parametrize("precision", [L.FP64, L.FP32, L.FP32_DEV, L.FP32_KAHAN, L.FP32_SPLIT, L.FP64_DW])
@pytest.mark.parametrize("nx,ny", [(3, 9001), (8, 70000), (260, 130), (1027, 1030), (2052, 901), (4100, 7)])
def test_device_transfers_equal_host_transfers(nx, ny, precision):
    import torch
    g = np.random.default_rng(nx)
    st = g.uniform(0, 1, (5, ny, nx))
    for dtype in (np.float32, np.float64):
        host = L.Solver(nx, ny, RATES, d=D, precision=precision)
        dev = L.Solver(nx, ny, RATES, d=D, precision=precision)
        host.write(st.astype(dtype))
        t = torch.from_numpy(st.astype(dtype)).cuda()
        dev.write(t)
        assert np.array_equal(dev.checkpoint()[128:], host.checkpoint()[128:])
        t.zero_()
        L.sslbm_read(dev.h, L.SCHEME_SSLBM, L.ALL, t)
        assert np.array_equal(t.cpu().numpy(), host.read(dtype=dtype))
        host.close()
        dev.close()
