"""The planner takes the kernels that the cases of tests/tile_cases.py are there to run (152
multiprocessors), among them passes of 16 steps and more; compiled on its own."""
import shutil
import subprocess

import pytest

from paper_2603_19789_gb300 import build

from tile_cases import CASES

CODE = r"""
#include <stdio.h>
#include "pass_plan.cuh"
using namespace sslbm;
int main() {
  long long lat, prec, bc, nx, ny, n;
  while (scanf("%lld %lld %lld %lld %lld %lld", &lat, &prec, &bc, &nx, &ny, &n) == 6) {
    const PassCost* c = pass_cost((int)lat, (int)prec, (int)bc);
    TilePlan p{0, 0};
    const bool t = tile_plan(*c, nx, ny, n, default_pass_depth(*c, nx, ny, 152), kAnyParity, 152, &p);
    const long long passes = t ? pass_count(n, p.depth, kAnyParity) : 1;
    printf("%d %d %lld\n", (int)t, p.nr, (n + passes - 1) / passes);
  }
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_the_cases_take_their_kernels(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(CODE)
    subprocess.run(["g++", "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, str(src), "-o", str(tmp_path / "t")],
                   check=True)
    inp = "".join(" ".join(map(str, c[:6])) + "\n" for c in CASES)
    out = subprocess.run([str(tmp_path / "t")], input=inp, check=True, capture_output=True, text=True).stdout.split("\n")
    depths = []
    for case, row in zip(CASES, out):
        tile, nr, depth = map(int, row.split())
        assert (tile, nr) == (1, case[6]), (case, row)
        depths.append(depth)
    assert max(depths) >= 20 and sum(d >= 16 for d in depths) >= 4
