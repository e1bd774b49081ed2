"""Which pointers passed as device memory the state transfers hand to a kernel: device memory of the
solver's own device at the values' alignment.  Host memory (pageable or pinned), managed memory,
memory of another device and odd addresses stay with the runtime's copies.  The rule is host code
(csrc/user_memory.cuh), compiled here on its own."""
import os
import shutil
import subprocess

import pytest

from paper_2603_19789_gb300 import build

CODE = r"""
#include <stdio.h>
#include "user_memory.cuh"
int main() {
  const cudaMemoryType types[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice,
                                  cudaMemoryTypeManaged};
  for (cudaMemoryType t : types)
    for (int dev = -1; dev < 2; ++dev)
      for (unsigned off = 0; off < 9; ++off)
        for (unsigned size = 4; size <= 8; size += 4)
          printf("%d %d %u %u %d\n", (int)t, dev, off, size, (int)sslbm::kernel_may_use(t, dev, 0, 0x10000 + off, size));
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_kernels_take_only_aligned_memory_of_their_own_device(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(CODE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-I", cuda, "-I", build.CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    rows = [tuple(map(int, r.split())) for r in subprocess.run([str(tmp_path / "t")], check=True, capture_output=True,
                                                                text=True).stdout.splitlines()]
    assert len(rows) == 4 * 3 * 9 * 2
    for kind, dev, off, size, ok in rows:
        assert bool(ok) == (kind == 2 and dev == 0 and off % size == 0), (kind, dev, off, size)
