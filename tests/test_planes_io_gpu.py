"""Device writes and reads of a state in one launch, aligned groups of four and odd widths, every
storage and value type, a single compartment, and buffers of odd alignment: the same values as
the host transfers, which go plane by plane; and the ensemble diagnostics, one launch for all."""
import numpy as np
import pytest

from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu

RATES = (0.5, 0.2, 0.11, 0.1)
D = (0.05, 0.04, 0.01, 0.05, 0.0)


@pytest.mark.parametrize("precision", [L.FP64, L.FP32, L.FP32_DEV, L.FP32_KAHAN, L.FP32_SPLIT, L.FP64_DW])
@pytest.mark.parametrize("nx,ny", [(1, 1), (4, 3), (512, 5), (516, 7), (513, 4), (1027, 2)])
def test_device_transfers_equal_host_transfers(nx, ny, precision):
    import torch
    st = inputs.epidemic_state(nx, ny, seed=nx)
    for dtype, tdtype in ((np.float32, torch.float32), (np.float64, torch.float64)):
        host = L.Solver(nx, ny, RATES, d=D, precision=precision)
        dev = L.Solver(nx, ny, RATES, d=D, precision=precision)
        host.write(st.astype(dtype))
        buf = torch.empty(5 * nx * ny + 1, dtype=tdtype, device="cuda")
        for off in (0, 1):  # off = 1: not 16-byte aligned
            t = buf[off:off + 5 * nx * ny].view(5, ny, nx)
            t.copy_(torch.from_numpy(st.astype(dtype)))
            dev.write(t)
            assert np.array_equal(dev.checkpoint()[128:], host.checkpoint()[128:])
            t.zero_()
            L.sslbm_read(dev.h, L.SCHEME_SSLBM, L.ALL, t)
            assert np.array_equal(t.cpu().numpy(), host.read(dtype=dtype))
        one = torch.full((ny, nx), 0.25, dtype=tdtype, device="cuda")
        for c in (L.S, L.I):
            dev.write(one, comp=c)
            host.write(one.cpu().numpy(), comp=c)
            got = torch.empty_like(one)
            L.sslbm_read(dev.h, L.SCHEME_SSLBM, c, got)
            assert np.array_equal(got.cpu().numpy(), host.read(comp=c, dtype=dtype))
        assert np.array_equal(dev.checkpoint()[128:], host.checkpoint()[128:])
        host.close()
        dev.close()


@pytest.mark.parametrize("precision", [L.FP32, L.FP32_DEV, L.FP32_SPLIT])
@pytest.mark.parametrize("n", [1, 3, 70])
def test_ensemble_diagnostics_of_all_scenarios(n, precision):
    """Every scenario's totals against an exact sum of what it reads back."""
    import math
    specs = [dict(nx=4 * (1 + i % 9), ny=1 + 5 * (i % 7), rates=RATES, d=D) for i in range(n)]
    ens = L.Ensemble(specs, precision=precision)
    for i, sp in enumerate(specs):
        ens.write(i, inputs.epidemic_state(sp["nx"], sp["ny"], seed=i))
    totals, peak = ens.diagnostics()
    for i in range(n):
        st = ens.read(i)
        want = [math.fsum(st[c].ravel()) for c in range(5)]
        np.testing.assert_allclose(totals[i], want, rtol=1e-12)
        assert peak[i] == st[2].max()
    ens.close()
