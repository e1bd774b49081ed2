"""How a call of n steps is cut into passes (csrc/pass_plan.cuh, host code, compiled here on its own):
every cut covers n with passes no deeper than allowed, and where a parity is asked for the number of
passes has it, for every n > 1."""
import shutil
import subprocess

import pytest

from paper_2603_19789_gb300 import build

CODE = r"""
#include <stdio.h>
#include "pass_plan.cuh"
using namespace sslbm;
int main() {
  for (int depth = 1; depth <= 8; ++depth)
    for (int deep = depth; deep <= 8; ++deep)
      for (int n = 1; n <= 130; ++n)
        for (int parity = -1; parity <= 1; ++parity) {
          int left = n, passes = 0, lo = 99, hi = 0, p = parity;
          while (left > 0) {
            const int k = next_pass_depth(left, depth, deep, p);
            p = flip_parity(p);
            left -= k, ++passes;
            lo = k < lo ? k : lo, hi = k > hi ? k : hi;
          }
          printf("%d %d %d %d %d %d %d %d %lld\n", depth, deep, n, parity, left, passes, lo, hi,
                 (long long)pass_count(n, depth, parity));
        }
  for (int n = 1; n < 40; ++n)
    printf("P %d %d %d %d %d\n", n, pass_parity(n, 4, false, false), pass_parity(n, 4, true, false),
           pass_parity(n, 4, true, true), pass_parity(n, 4, false, true));
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_cuts_cover_n_with_the_parity_asked_for(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(CODE)
    subprocess.run(["g++", "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, str(src), "-o", str(tmp_path / "t")],
                   check=True)
    out = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(out) == 36 * 130 * 3 + 39
    for row in out:
        if row[0] == "P":
            n, free, cap, again, after = map(int, row.split()[1:])
            assert (free, cap, again, after) == (-1, 0, 0, -(-n // 4) % 2)
            continue
        depth, deep, n, parity, left, passes, lo, hi, count = map(int, row.split())
        what = (depth, deep, n, parity)
        assert left == 0 and 1 <= lo and hi <= deep, what
        if parity >= 0 and n > 1 and depth > 1:
            assert passes % 2 == count % 2 == parity, what
        if parity < 0 and deep == depth:
            assert passes == count == -(-n // depth) and hi - lo <= 1, what
