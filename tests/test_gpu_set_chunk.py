"""A chunk length the caller sets on the float32 shape 56 x 28: it stays the one reported, items are never longer and
at least half as long, and they are shorter only where the set length would leave the GPU's last round of items nearly
empty. The fields are the same bits for every length (the same operations in the same order)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_0901_1053_gb300 import workloads as wl  # noqa: E402


@pytest.fixture(scope="module")
def tetm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_0901_1053_gb300 import tetm as t
    return t


def rounds(items):
    return math.ceil(items / (2 * torch.cuda.get_device_properties(0).multi_processor_count))


# 2 x 19 tiles: 9 chunks of 32 planes are just more items than the GPU holds at once, 8 just fewer; a chunk of one
# plane's remainder, the shortest, longer than the grid
@pytest.mark.parametrize("nz,cz", [(257, 32), (256, 32), (40, 7), (130, 4), (130, 5), (90, 200), (2, 4)])
def test_set_chunk(tetm, nz, cz):
    nx, ny = 112, 228
    tiles = 38
    s = tetm.Solver(nx, ny, nz, wl.DXY, wl.DXY, wl.DZ, wl.DZ, "fp32")
    s.set_tiling(56, 28, cz)
    info = s.info()
    assert (info["tile_x"], info["tile_y"], info["chunk_z"]) == (56, 28, cz)
    chunks = info["work_items"] // tiles
    assert info["work_items"] == tiles * chunks
    longest = min(cz, nz)
    assert math.ceil(nz / longest) <= chunks <= math.ceil(nz / max(4, math.ceil(longest / 2)))
    # by the cost of a step, rounds of the GPU times planes and two more, no length between the half and the whole is
    # more than a ninth cheaper (an item's length is no less than ceil(nz / chunks))
    cost = rounds(info["work_items"]) * (math.ceil(nz / chunks) + 2)
    least = min(rounds(tiles * math.ceil(nz / c)) * (c + 2) for c in range(min(max(4, math.ceil(longest / 2)), longest), longest + 1))
    assert cost <= least / 0.9
    if (nz, cz) == (256, 32):
        assert chunks == 8            # a whole round as set
    out = []
    for other in (False, True):
        if other:
            s.close()
            s = tetm.Solver(nx, ny, nz, wl.DXY, wl.DXY, wl.DZ, wl.DZ, "fp32")
            s.set_tiling(28, 20, 16)
        s.set_bunch(2.3 * wl.DZ, 1e-9, nx // 2, ny // 2)
        for c, a in enumerate(wl.random_fields(s.shape, 7)):
            s.set(c, a)
        s.step(5)
        out.append([s.get(c) for c in range(6)])
        assert s.check_guards() == 0
    s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_a_batch_takes_the_set_length(tetm):
    members, want = [], []
    for k in range(2):
        s = tetm.Solver(112, 228, 257, wl.DXY, wl.DXY, wl.DZ, wl.DZ, "fp32")
        s.set_tiling(56, 28, 32)
        s.set_bunch(2.3 * wl.DZ, 1e-9, 56, 114)
        members.append(s)
    ref = tetm.Solver(112, 228, 257, wl.DXY, wl.DXY, wl.DZ, wl.DZ, "fp32")
    ref.set_bunch(2.3 * wl.DZ, 1e-9, 56, 114)
    ref.step(20)
    b = tetm.Batch(members, [20, 20], graph_steps=4)
    assert b.info()["work_items"] == 2 * 38 * 9
    b.step(20)
    b.sync()
    b.close()
    for s in members:
        for c in range(6):
            assert np.array_equal(s.get(c), ref.get(c))
        s.close()
    ref.close()
