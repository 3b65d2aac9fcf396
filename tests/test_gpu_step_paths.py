"""Which step a solve takes, seen in tetm_get_info's processed_cells (the cells that the items of its step own), and
the branches of that choice at the sizes where each begins and ends.

Tolerance: none for fields and wakes, the paths do the same operations per node in the same order and round every
wake sample alike; where samples are summed by several items the order is free: n additions of one rounding each."""
import math

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


def cartesian(tetm, dims, precision, pec=None, tiling=None, eps=None):
    nx, ny, nz = dims
    s = tetm.Solver(nx, ny, nz, wl.DXY, wl.DXY, wl.DZ, wl.DZ, precision, pec=pec, eps_r=eps)
    if tiling:
        s.set_tiling(*tiling)
    s.set_bunch(2.3 * wl.DZ, 1e-9, nx // 2, ny // 2)
    s.set_observer(nx // 2, ny // 2)
    return s


def run(s, steps=3):
    rng = np.random.default_rng(11)
    f = rng.standard_normal(s.shape)
    for c in range(6):
        s.set(c, np.roll(f, 7 * c + 1, axis=2))
    s.step(steps)
    out = [s.get(c) for c in range(6)], [s.wake()[0], *s.transverse_wake()]
    assert s.check_guards() == 0
    s.close()
    return out


def same(a, b, nz):
    for x, y in zip(a[0], b[0]):
        assert np.array_equal(x, y)
    for x, y in zip(a[1], b[1]):
        assert np.abs(x - y).max() <= 4 * nz * np.finfo(float).eps * max(np.abs(y).max(), 1e-300)


# float64: from 2 << 20 active cells on the bands have 16 rows instead of 8. An open box's items own every cell, so
# the two cannot be told apart there; with one wall row in eight (of sixteen) only whole bands disappear.
@pytest.mark.parametrize("dims,rows", [((130, 130, 124), 8), ((130, 130, 134), 16), ((129, 133, 140), 16)])
def test_float64_bands(tetm, dims, rows):
    nx, ny, nz = dims
    pec = np.zeros((nz, ny, nx), np.uint8)
    pec[:, 16:24, :] = 1                       # a band of 8 rows in PEC, half a band of 16
    s = cartesian(tetm, dims, "fp64", pec)
    info = s.info()
    assert (info["active_cells"] >= 2 << 20) == (rows == 16)
    owned = sum(min(rows, ny - j) for j in range(0, ny, rows) if not pec[0, j:j + rows, 0].all())
    assert info["processed_cells"] == owned * nx * nz
    assert (info["tile_x"], info["tile_y"], info["chunk_z"]) == (28, 20, 32)
    w = cartesian(tetm, dims, "fp64", pec, (28, 20, 32))
    assert w.info()["processed_cells"] == w.info()["work_items"] * 28 * 20 * 32
    same(run(s), run(w), nz)


# float32: half-steps up to 3 << 18 active cells, in runs of planes; beyond, the sweep. (116, 52, 129) is just below,
# (116, 53, 129) just above; runs of one plane on the smallest.
@pytest.mark.parametrize("dims,half", [((2, 2, 2), True), ((57, 15, 9), True), ((116, 52, 130), True),
                                       ((116, 53, 129), False)])
def test_float32_half_steps(tetm, dims, half):
    nx, ny, nz = dims
    s = cartesian(tetm, dims, "fp32")
    info = s.info()
    assert info["active_cells"] == nx * ny * nz - 1            # every entry of node (0, 0, 0) lies on a wall
    assert (info["active_cells"] <= 3 << 18) == half
    tiles = math.ceil(nx / 56) * math.ceil(ny / 14)
    runs = [tiles * math.ceil(nz / r) * 56 * 14 * r for r in range(1, 9)]
    slab = info["work_items"] * 56 * 12 * info["chunk_z"]
    assert info["processed_cells"] in (runs if half else [slab])
    assert not half or info["processed_cells"] != slab
    t = cartesian(tetm, dims, "fp32", tiling=(0, 0, 5))
    # (items of the set length, or of four planes where five leave the GPU emptier)
    assert t.info()["processed_cells"] in [t.info()["work_items"] * 56 * 12 * z for z in (4, 5)]
    same(run(s), run(t), nz)


def test_a_batch_member_reports_its_items(tetm):
    s = cartesian(tetm, (57, 15, 9), "fp32")
    alone = s.info()["processed_cells"]
    b = tetm.Batch([s], [4])
    i = s.info()
    assert i["processed_cells"] == i["work_items"] * 56 * 12 * i["chunk_z"]
    b.step(4)
    b.close()
    assert s.info()["processed_cells"] == alone
    s.close()


def test_batch_work_items_are_those_still_stepped(tetm):
    """(member, item) entries of the members below their limit, before and after members retire, join and leave."""
    dims = [(64, 64, 130), (57, 13, 5), (113, 25, 67)]
    for tile in ((56, 28), (28, 20)):
        b = tetm.Batch.slots(3, "fp32", tile, graph_steps=2)
        assert b.info()["work_items"] == 0
        per = {}
        members = []
        for d, limit in zip(dims, (2, 5, 9)):
            s = cartesian(tetm, d, "fp32")
            before = b.info()["work_items"]
            b.add(s, limit)
            per[limit] = b.info()["work_items"] - before
            members.append(s)
        assert all(per.values())
        for step in range(1, 11):
            b.step(1)
            assert b.info()["work_items"] == sum(n for limit, n in per.items() if step < limit)
        extra = cartesian(tetm, dims[0], "fp32")
        b.remove(members[0])
        b.add(extra, 3)
        assert b.info()["work_items"] == per[2]
        b.remove(extra)
        assert b.info()["work_items"] == 0
        b.sync()
        b.close()


def test_rz_reports_the_kernel_that_steps(tetm):
    pec = wl.cavity_chain_rz(57, 70, 0, 1).pec
    cells = int((pec == 0).sum())
    f = tetm.RzSolver(57, 70, 0, 1, 1e-3, 1e-3, 1e-3, "fp32", pec=pec)
    assert f.info()["kernel"] == tetm.TETM_RZ_KERNEL_BULK2
    f.set_kernel("async")
    assert f.info()["kernel"] == tetm.TETM_RZ_KERNEL_ASYNC
    d = tetm.RzSolver(57, 70, 0, 1, 1e-3, 1e-3, 1e-3, "fp64", pec=pec)
    bands = d.info()["processed_cells"]
    assert 2 * cells <= bands < 2 * 58 * 70     # the runs cover the open columns, not the walls
    d.set_kernel("async")
    assert d.info()["processed_cells"] != bands and d.info()["kernel"] == tetm.TETM_RZ_KERNEL_ASYNC
