"""Every register-tile kernel that the default blocking takes (tests/tile_cases.py): the bits of one step per
launch, and in the index-checked build no index out of range."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2603_19789_gb300 import build, inputs
from paper_2603_19789_gb300 import sslbm as L

from tile_cases import CASES

pytestmark = pytest.mark.gpu

RATES = (0.5, 0.2, 0.11, 0.1)
D = (0.05, 0.04, 0.01, 0.05, 0.0)
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _solver(lattice, precision, bc, nx, ny):
    s = L.Solver(nx, ny, RATES, d=D, bc=bc, precision=precision, lattice=lattice)
    if lattice == L.LATTICE_D2Q5_VARD:
        s.set_diffusivity_scale(*inputs.mobility_fields(nx, ny, seed=3, kind="random"))
    s.write(inputs.epidemic_state(nx, ny, seed=nx + 7 * ny))
    return s


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_tile_kernels_give_the_bits_of_one_step_launches(case):
    lattice, precision, bc, nx, ny, n, _ = case
    s, ref = _solver(lattice, precision, bc, nx, ny), _solver(lattice, precision, bc, nx, ny)
    ref.set_blocking(1)
    s.step(n)
    ref.step(n)
    a, b = s.read(dtype=np.float32), ref.read(dtype=np.float32)
    assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
    s.close()
    ref.close()


SWEEP = r"""
import json, sys
sys.path.insert(0, "tests")
from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L
from tile_cases import CASES
L.load()
runs = 0
tiny = [c[:3] + (nx, ny, n) for c in CASES[::4] for nx, ny in ((1, 1), (2, 7), (5, 1), (31, 64), (65, 130), (130, 67)) for n in (2, 13, 29)]
for lattice, precision, bc, nx, ny, n in [c[:6] for c in CASES] + tiny:
    s = L.Solver(nx, ny, (0.5, 0.2, 0.11, 0.1), d=(0.05, 0.04, 0.01, 0.05, 0.0), bc=bc, precision=precision, lattice=lattice)
    if lattice == L.LATTICE_D2Q5_VARD:
        s.set_diffusivity_scale(*inputs.mobility_fields(nx, ny, seed=3, kind="random"))
    s.write(inputs.epidemic_state(nx, ny, seed=nx + 7 * ny))
    s.step(n)
    s.read()
    s.close()
    runs += 1
for bc in (L.BC_PERIODIC, L.BC_NOFLUX):
    for nx, ny in ((1, 1), (3, 2), (61, 33), (130, 67), (700, 300)):
        s = L.Solver(nx, ny, (0.5, 0.2, 0.11, 0.1), d=(0.05, 0.04, 0.01, 0.05, 0.0), bc=bc, precision=L.FP32, schemes=L.WANT_BGK)
        s.write(inputs.epidemic_state(nx, ny, seed=nx + ny), scheme=L.SCHEME_BGK)
        for n in (2, 3, 4, 7):
            s.bgk_step(n)
        s.close()
        runs += 1
print(json.dumps(dict(runs=runs, bounds=L.sslbm_debug_bounds())))
"""


def test_tile_kernels_stay_in_bounds():
    lib = build.build(checked=True)
    r = subprocess.run([sys.executable, "-c", SWEEP], capture_output=True, text=True, cwd=ROOT,
                       env={**os.environ, "SSLBM_LIBRARY": lib})
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.splitlines()[-1])
    assert out["runs"] == len(CASES) + 6 * 3 * len(CASES[::4]) + 10
    assert out["bounds"]["count"] == 0, out
