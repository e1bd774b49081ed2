"""Grids and step counts that take each register-tile kernel under the default blocking on a GPU of 152
multiprocessors: (lattice, storage, boundary, nx, ny, steps, rows per warp, depth of the deepest pass).
tests/test_tile_cases_cpu.py holds the planner to them, tests/test_tile_cases_gpu.py runs them."""
from paper_2603_19789_gb300 import sslbm as L

D5, D9, VD = L.LATTICE_D2Q5, L.LATTICE_D2Q9, L.LATTICE_D2Q5_VARD
PER, WALL = L.BC_PERIODIC, L.BC_NOFLUX

CASES = []
for lattice, precision in ((D5, L.FP32), (D5, L.FP32_DEV), (D9, L.FP32), (VD, L.FP32)):
    for bc in (PER, WALL):
        CASES += [(lattice, precision, bc, nx, ny, n, 4) for nx, ny, n in ((513, 517, 23), (1001, 777, 21), (1023, 900, 16))]
        CASES += [(lattice, precision, bc, 200, 100, 60, 1)]
CASES += [(D5, L.FP32, WALL, 1, 1, 100, 2), (D5, L.FP32_DEV, PER, 300, 200, 40, 2), (D9, L.FP32, PER, 300, 200, 40, 2),
          # the deepest passes that the planner takes anywhere
          (D5, L.FP32, WALL, 1, 2749, 400, 4), (D9, L.FP32, PER, 56, 1783, 400, 4), (D9, L.FP32, WALL, 62, 2120, 16, 4),
          (VD, L.FP32, WALL, 62, 2120, 16, 4)]
