"""A float32 batch whose members reach their limits at different steps: the items of retired members leave the work
list, the others' fields are the same bits as alone (no tolerance: the same operations in the same order)."""
import numpy as np
import pytest

from paper_0901_1053_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tetm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_0901_1053_gb300 import tetm as t
    return t


def solver(tetm, dims, cz):
    nx, ny, nz = dims
    s = tetm.Solver(nx, ny, nz, wl.DXY, wl.DXY, wl.DZ, wl.DZ, "fp32")
    s.set_tiling(0, 0, cz)
    s.set_bunch(2.3 * wl.DZ, 1e-9, nx // 2, ny // 2)
    for c, a in enumerate(wl.random_fields(s.shape, nx + nz)):
        s.set(c, a)
    return s


# fewer items than the compacting block has threads, and several times as many; retiring first, last and in between,
# two at once, all at once
@pytest.mark.parametrize("cz", [4, 64])
@pytest.mark.parametrize("limits", [(3, 5, 5, 9, 12, 12), (12, 9, 5, 5, 3, 1), (4, 4, 4, 4, 4, 4)])
def test_members_retire(tetm, cz, limits):
    dims = [(64, 64, 130), (57, 13, 5), (113, 25, 67), (64, 64, 130), (2, 2, 2), (80, 40, 90)]
    members = [solver(tetm, d, cz) for d in dims]
    b = tetm.Batch(members, list(limits), graph_steps=4)
    b.step(max(limits))
    b.sync()
    b.close()
    for d, n, m in zip(dims, limits, members):
        s = solver(tetm, d, cz)
        s.step(n)
        assert m.info()["step"] == n
        for c in range(6):
            assert np.array_equal(s.get(c), m.get(c))
        s.close()
        m.close()
