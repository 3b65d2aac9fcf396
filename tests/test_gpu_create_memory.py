"""A float64 solve with material arrays needs no more device memory while it is made than when it is there: the cell
arrays on the device are released before the last of its own arrays are allocated. The allocating source is compiled
once more with its allocations counted, and linked with the other objects."""
import glob
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = """
#include <cuda_runtime.h>
#include <map>
extern "C" { __attribute__((visibility("default"))) long long held = 0, peak = 0; }
static std::map<void*, size_t> sizes;
static inline cudaError_t counted(void** p, size_t bytes, cudaMemPool_t pool, cudaStream_t st) {
  cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, st);
  if (e == cudaSuccess) {
    sizes[*p] = bytes;
    held += (long long)bytes;
    if (held > peak) peak = held;
  }
  return e;
}
static inline cudaError_t released(void* p, cudaStream_t st) {
  held -= (long long)sizes[p];
  sizes.erase(p);
  return cudaFreeAsync(p, st);
}
#define cudaMallocFromPoolAsync counted
#define cudaFreeAsync released
"""

CHILD = """
import ctypes, sys
sys.path.insert(0, %(root)r)
from paper_0901_1053_gb300 import build
build.library_path = lambda: %(lib)r
from paper_0901_1053_gb300 import tetm, workloads as wl

held = ctypes.c_longlong.in_dll(tetm.lib, "held")
peak = ctypes.c_longlong.in_dll(tetm.lib, "peak")
nx, ny, nz = 64, 48, 80
eps, mu, pec = wl.random_materials(nx, ny, nz, 3)
for a, b in ((eps, None), (eps, mu)):
    peak.value = 0
    s = tetm.Solver(nx, ny, nz, wl.DXY, wl.DXY, wl.DZ, wl.DZ, "fp64", pec=pec, eps_r=a, mu_r=b)
    assert held.value >= 240 * nx * ny * nz
    assert peak.value <= held.value, (peak.value, held.value)
    s.close()
    assert held.value == 0
print("no more")
"""


def test_creation_needs_no_more_than_the_solve(tmp_path):
    import __graft_entry__
    __graft_entry__.build()
    from paper_0901_1053_gb300 import build
    (tmp_path / "shim.h").write_text(SHIM)
    obj, lib = str(tmp_path / "counted.o"), str(tmp_path / "libtetm_counted.so")
    common = [build.nvcc()] + build.ARCH
    subprocess.run(common + build.NVCC_FLAGS + ["-include", str(tmp_path / "shim.h"), "-c",
                   os.path.join(build.CSRC, "capi.cu"), "-o", obj], check=True)
    others = [o for o in sorted(glob.glob(os.path.join(build.BUILD_DIR, "*.o"))) if not o.endswith("/capi.o")]
    subprocess.run(common + ["-shared", "-o", lib, obj] + others + ["-lcuda"], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT, "lib": lib}], capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0 and "no more" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
