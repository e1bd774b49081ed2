"""Kernels that may start before their predecessor ends (they call pdl_enter) read memory only after
that call: none takes a __restrict__ pointer, which would let the compiler read through it earlier or
through the read-only path.  The row pipeline, whose global reads are cp.async in volatile assembly,
is the exception."""
import glob
import os
import re

from paper_2603_19789_gb300 import build

CP_ASYNC_ONLY = {"pipe_kernel"}


def _kernels():
    for path in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))):
        text = open(path).read()
        heads = list(re.finditer(r"__global__ void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(([^)]*)\)", text))
        for m, nxt in zip(heads, heads[1:] + [None]):
            body = text[m.end():nxt.start() if nxt else len(text)]
            yield os.path.basename(path), m.group(1), m.group(2), body


def test_dependent_kernels_take_no_restrict_pointers():
    dependent = {name: (path, params) for path, name, params, body in _kernels() if re.search(r"\bpdl_enter\(\);", body)}
    assert {"tile_kernel", "bgk_tile_kernel", "planes_io_kernel", "step1_kernel", "fd4_pair_kernel",
            "stream_kernel", "pipe_kernel"} <= set(dependent)
    for name, (path, params) in dependent.items():
        if name not in CP_ASYNC_ONLY:
            assert "__restrict__" not in params, (path, name)
