"""The ensemble's workspace is its two state buffers and a fixed amount per scenario: the diagnostics'
partial sums take no room that grows with the grids' rows."""
import pytest

from paper_2603_19789_gb300 import sslbm as L

RATES = (0.5, 0.2, 0.11, 0.1)
D = (0.05, 0.04, 0.01, 0.05, 0.0)


@pytest.mark.parametrize("precision,planes", [(L.FP32, 5), (L.FP32_DEV, 5), (L.FP32_SPLIT, 6)])
@pytest.mark.parametrize("n,nx,ny", [(1, 4, 1), (32, 1024, 1024), (32, 64, 4096), (3, 512, 16384)])
def test_workspace_beyond_the_states_is_fixed_per_scenario(n, nx, ny, precision, planes):
    sc = L.make_scenarios([dict(nx=nx, ny=ny, rates=RATES, d=D)] * n)
    plane = (-(-nx // 32) * 32 * ny + 63) // 64 * 64
    states = 2 * (-(-(n * planes * plane * 4) // 256) * 256)
    # control words, counters, table, results, and the 48 KiB that one grid's partial sums take
    assert 0 < L.sslbm_ensemble_workspace_bytes(sc, precision) - states <= 49152 + 4 * 256 + n * (4 + 160 + 48)
