"""Launches that are split by rows when no memory can be had for it: the library
is linked with a cudaMalloc that refuses, and rows and checksums still come out,
without bands.  In a process of its own, since the library is another one."""
import os
import subprocess
import sys

import pytest

from paper_1609_01257_gb300 import builder

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

WRAP = """
#include <cuda_runtime_api.h>
extern "C" { int refuse_malloc = 0; }
extern "C" cudaError_t __real_cudaMalloc(void **p, size_t bytes);
extern "C" cudaError_t __wrap_cudaMalloc(void **p, size_t bytes) {
  return refuse_malloc ? cudaErrorMemoryAllocation : __real_cudaMalloc(p, bytes);
}
"""

CHILD = """
import ctypes, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
from paper_1609_01257_gb300 import builder
builder.LIB = sys.argv[2]
import oracle
import paper_1609_01257_gb300 as rng

refuse = ctypes.c_int.in_dll(rng.load(), "refuse_malloc")
for n, T, mode in [(65_536, 300, 0), (1001, 700, 1), (1_300_001, 200, 1), (8192, 17_000, 0)]:
    for states in (False, True):
        g = rng.Generator(n, 83, output_mode=mode)
        p = 0
        if states:
            g.skip(7)
            p = 7
        refuse.value = 1
        x, s = (v.cpu().numpy() for v in g.generate_checksum(T))
        rows = g.generate(min(T, 260)).cpu().numpy()
        band_rows = g.last_launch()["band_rows"]
        refuse.value = 0
        g.close()
        wx, ws, _ = oracle.row_checksums(n, 83, T, p0=p, output_mode=mode)
        assert np.array_equal(x, wx) and np.array_equal(s, ws), (n, states)
        assert np.array_equal(rows, oracle.generate(n, 83, len(rows), p0=p + T, output_mode=mode)), (n, states)
        assert band_rows == 0
print("no memory: ok")
"""


def test_no_memory_for_bands(tmp_path):
    objs = [os.path.join(builder.BUILD, "obj", os.path.basename(s) + ".o") for s in builder.sources()]
    if not all(os.path.exists(o) for o in objs):
        builder.build(force=True)
    src, lib = tmp_path / "wrap.cpp", tmp_path / "librng_wrapped.so"
    src.write_text(WRAP)
    subprocess.run([builder._nvcc(), *builder.ARCH, "-shared", "-cudart", "static", "-Xcompiler", "-fPIC",
                    "-Xlinker", "--wrap=cudaMalloc", "-o", str(lib), str(src), *objs, "-lpthread"],
                   check=True, timeout=300)
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(lib)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "no memory: ok" in r.stdout, r.stdout + r.stderr
