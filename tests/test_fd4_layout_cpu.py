"""The finite-difference reference's workspace: four states of five contiguous planes [5][ny][nx], each
rounded up to 256 bytes, whatever the width and the precision."""
import pytest

from paper_2603_19789_gb300 import sslbm as L


@pytest.mark.parametrize("precision,size", [(L.FP32, 4), (L.FP64, 8)])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 50), (127, 64), (128, 64), (201, 199), (1001, 777)])
def test_workspace_is_four_contiguous_states(nx, ny, precision, size):
    grid = L.make_grid(nx, ny, 1.0, 0.25, L.BC_NOFLUX, precision)
    assert L.sslbm_fd4_workspace_bytes(grid) == 4 * ((5 * nx * ny * size + 255) // 256 * 256)
