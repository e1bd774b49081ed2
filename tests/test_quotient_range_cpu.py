"""The integer steps of the FP64 quotient (csrc/quot_range.cuh, compiled here with the undefined-behaviour
sanitizer): the range test agrees with the values on every kind of divisor -- zeros, negatives down to
the smallest, infinities, NaN, both ends of the range -- and the float's bits become its double."""
import shutil
import subprocess

import pytest

from paper_2603_19789_gb300 import build

CODE = r"""
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
#include "quot_range.cuh"
static int hi(double d) { uint64_t u; memcpy(&u, &d, 8); return (int)(uint32_t)(u >> 32); }
int main() {
  const double v[] = {0.0, -0.0, 5e-324, -5e-324, 1e-310, -1e-310, ldexp(1, -99), nextafter(ldexp(1, -99), 0), -ldexp(1, -99),
                      1.0, -1.0, 125.0, nextafter(ldexp(1, 99), 0), ldexp(1, 99), 1e308, -1e308, INFINITY, -INFINITY, NAN, -NAN};
  for (double d : v) {
    const bool want = d >= ldexp(1, -99) && d < ldexp(1, 99);
    if (sslbm::quot_in_range(hi(d)) != want) return printf("range %g\n", d), 1;
  }
  for (int e = -99; e <= 99; ++e)
    for (uint32_t m = 0; m < (1u << 23); m += 524287) {
      const uint32_t rb = (uint32_t)(e + 127) << 23 | m;
      float f; memcpy(&f, &rb, 4);
      const uint64_t u = (uint64_t)(uint32_t)sslbm::quot_hi((int)rb) << 32 | (uint32_t)sslbm::quot_lo((int)rb);
      double d; memcpy(&d, &u, 8);
      if (d != (double)f) return printf("value %g %g\n", d, f), 1;
    }
  puts("ok");
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_range_and_format_change(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(CODE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-I", build.CSRC,
                    str(src), "-o", str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr
