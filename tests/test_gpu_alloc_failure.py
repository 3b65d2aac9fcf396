"""Device memory that runs out while a solve takes another work shape: the call
answers TETM_E_NOMEM and the solve keeps its shape, its item list and its
results. A list read under another tile shape would send a kernel past the
grid, so nothing is stepped before the reported shape has been checked.

The failure is made on the host: the allocating source is compiled once more
with the allocation call replaced by one that answers
cudaErrorMemoryAllocation at a chosen call, and linked with the other objects."""
import glob
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = """
#include <cuda_runtime.h>
extern "C" { __attribute__((visibility("default"))) int fail_alloc_at = 0; }  // 1: the next one, 0: none
static inline cudaError_t alloc_or_fail(void** p, size_t bytes, cudaMemPool_t pool, cudaStream_t st) {
  if (fail_alloc_at > 0 && --fail_alloc_at == 0) return cudaErrorMemoryAllocation;
  return cudaMallocFromPoolAsync(p, bytes, pool, st);
}
#define cudaMallocFromPoolAsync alloc_or_fail
"""

CHILD = """
import ctypes, sys
sys.path.insert(0, %(root)r)
from paper_0901_1053_gb300 import build
build.library_path = lambda: %(lib)r
import numpy as np
from paper_0901_1053_gb300 import tetm, workloads as wl

fail = ctypes.c_int.in_dll(tetm.lib, "fail_alloc_at")
SHAPE = ("tile_x", "tile_y", "chunk_z", "work_items", "processed_cells")
NX, NY, NZ = 64, 64, 130

def solver(precision, eps=None):
    s = tetm.Solver(NX, NY, NZ, wl.DXY, wl.DXY, wl.DZ, wl.DZ, precision, eps_r=eps)
    s.set_bunch(2.3 * wl.DZ, 1e-9, NX // 2, NY // 2)
    for c, a in enumerate(wl.random_fields(s.shape, 5)):
        s.set(c, a)
    return s

def shape(s):
    return [s.info()[k] for k in SHAPE]

def refused(call, s):
    # one refusal per allocation of the call, then the call itself
    before, n = shape(s), 0
    while True:
        n += 1
        fail.value = n
        try:
            call()
        except tetm.TetmError as e:
            assert e.code == tetm.TETM_E_NOMEM, e.code
            assert shape(s) == before, (shape(s), before)
        else:
            assert fail.value > 0        # no allocation was left to refuse
            fail.value = 0
            return n - 1

def same(a, b):
    for c in range(6):
        assert np.array_equal(a.get(c), b.get(c))
    assert a.energy() == b.energy()

eps = np.random.default_rng(1).uniform(1.0, 3.0, size=(NZ, NY, NX))
for precision, e, tiling in (("fp32", None, (28, 4, 4)), ("fp64", None, (28, 4, 4)), ("fp32", eps, (28, 8, 4))):
    s, want = solver(precision, e), solver(precision, e)
    n0 = shape(s)
    fail.value = 1
    try:
        s.set_tiling(*tiling)
        raise SystemExit("accepted without memory")
    except tetm.TetmError:
        assert shape(s) == n0, (shape(s), n0)
    s.step(3)                            # on the shape it had, the library's choice
    want.step(3)
    same(s, want)
    assert refused(lambda: s.set_tiling(*tiling), s) == 3   # tile planes, partials, list
    s.step(2)
    want.set_tiling(*tiling)
    want.step(2)
    same(s, want)
    s.close()
    want.close()

s = solver("fp32")                       # a scheme switch that fails leaves the scheme
t = tetm.Solver(NX, NY, NZ, wl.DXY, wl.DXY, wl.DZ, 0.5 * wl.DZ, "fp32")
assert refused(lambda: t.set_scheme("yee"), t) >= 2
t.close()

want = solver("fp32")                    # so does a batch that cannot take the member
b = tetm.Batch.slots(2, "fp32", (28, 20))
assert refused(lambda: b.add(s, 3), s) >= 2
b.step(3)
b.sync()
b.remove(s)
want.step(3)
for c in range(6):
    assert np.array_equal(s.get(c), want.get(c))
b.close()

n = 0                                    # a solve that cannot be made: an error, whatever the allocation
for precision, e in (("fp32", None), ("fp32", eps), ("fp64", None), ("fp64", eps)):
    for n in range(1, 100):
        fail.value = n
        try:
            solver(precision, e).close()
        except tetm.TetmError:
            continue
        if fail.value > 0:               # none was left to refuse (a refused check of eps_r is done on the host)
            break
    assert 10 < n < 99, n
    fail.value = 0
s.step(2)                                # and the others go on
want.step(2)
for c in range(6):
    assert np.array_equal(s.get(c), want.get(c))
print("all kept")
"""


RZ_SHIM = """
#include <cuda_runtime.h>
extern "C" { __attribute__((visibility("default"))) int fail_alloc_at = 0; }  // 1: the next one, 0: none
template <typename P>
static inline cudaError_t alloc_or_fail(P* p, size_t bytes) {
  if (fail_alloc_at > 0 && --fail_alloc_at == 0) return cudaErrorMemoryAllocation;
  return cudaMalloc(p, bytes);
}
#define cudaMalloc alloc_or_fail
"""

RZ_CHILD = """
import ctypes, sys
sys.path.insert(0, %(root)r)
from paper_0901_1053_gb300 import build
build.library_path = lambda: %(lib)r
import numpy as np
from paper_0901_1053_gb300 import tetm, workloads as wl

fail = ctypes.c_int.in_dll(tetm.lib, "fail_alloc_at")
SHAPE = ("chunk_z", "work_items", "processed_cells", "resident_warps", "kernel")
NR, NZ = 130, 90
pec = wl.cavity_chain_rz(NR, NZ, 0, 2).pec

def solver(precision):
    s = tetm.RzSolver(NR, NZ, 0, 1, 1e-3, 1e-3, 1e-3, precision, pec=pec)
    rng = np.random.default_rng(3)
    for m in (0, 1):
        for c in range(6):
            s.set(m, c, rng.standard_normal(s.shape))
    return s

def shape(s):
    return [s.info()[k] for k in SHAPE]

def refused(call, s):
    before, n = shape(s), 0
    while True:
        n += 1
        fail.value = n
        try:
            call()
        except tetm.TetmError as e:
            assert e.code == tetm.TETM_E_NOMEM, e.code
            assert shape(s) == before, (shape(s), before)
        else:
            assert fail.value > 0
            fail.value = 0
            return n - 1

def same(a, b):
    for m in (0, 1):
        for c in range(6):
            assert np.array_equal(a.get(m, c), b.get(m, c))

for precision in ("fp32", "fp64"):
    s, want = solver(precision), solver(precision)
    n0 = shape(s)
    fail.value = 1
    try:
        s.set_kernel("bulk")
        raise SystemExit("accepted without memory")
    except tetm.TetmError:
        assert shape(s) == n0, (shape(s), n0)
    s.step(3)                            # on the library's choice
    want.step(3)
    same(s, want)
    for kernel, chunk in (("bulk", 5), ("bulk2", 4), ("register", 90)):
        assert refused(lambda: s.set_kernel(kernel), s) <= 2
        assert refused(lambda: s.set_tiling(chunk), s) >= 1
        s.step(3)
        want.step(3)
        same(s, want)
    s.close()
    want.close()
    for n in range(1, 100):              # a solve that cannot be made: an error, whatever the allocation
        fail.value = n
        try:
            solver(precision).close()
        except tetm.TetmError:
            continue
        break
    assert 8 < n < 99 and fail.value > 0, n
    fail.value = 0
print("all kept")
"""


@pytest.mark.parametrize("source,shim,child", [("capi.cu", SHIM, CHILD), ("rz.cu", RZ_SHIM, RZ_CHILD)],
                         ids=["cartesian", "rz"])
def test_a_failed_change_of_shape_changes_nothing(tmp_path, source, shim, child):
    import __graft_entry__
    __graft_entry__.build()
    from paper_0901_1053_gb300 import build
    (tmp_path / "shim.h").write_text(shim)
    obj, lib = str(tmp_path / "failing.o"), str(tmp_path / "libtetm_failing.so")
    common = [build.nvcc()] + build.ARCH
    subprocess.run(common + build.NVCC_FLAGS + ["-include", str(tmp_path / "shim.h"), "-c",
                   os.path.join(build.CSRC, source), "-o", obj], check=True)
    others = [o for o in sorted(glob.glob(os.path.join(build.BUILD_DIR, "*.o")))
              if os.path.basename(o) != source[:-3] + ".o"]
    subprocess.run(common + ["-shared", "-o", lib, obj] + others + ["-lcuda"], check=True)
    r = subprocess.run([sys.executable, "-c", child % {"root": ROOT, "lib": lib}], capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0 and "all kept" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
