"""The float32 slab kernel's work items: 56 x 12 nodes and, until the caller
sets a chunk, a number of planes chosen for the geometry. The fields are the
same bits for every length, alone and in a batch; the items are those that own
a field-carrying cell."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_0901_1053_gb300 import tetm, workloads as wl  # noqa: E402

COMPS = ("ex", "ey", "ez", "hx", "hy", "hz")


def build(n, kind, seed=5):
    nx, ny, nz = n
    rs = np.random.default_rng(seed)
    pec = eps = None
    if kind != "box":
        pec = (rs.uniform(size=(nz, ny, nx)) < 0.2).astype(np.uint8)
        pec[nz // 2:] |= (np.abs(np.arange(ny) - ny // 2) > ny // 3).astype(np.uint8)[:, None]
    if kind == "mat":
        eps = rs.uniform(1.0, 3.0, size=(nz, ny, nx))
    s = tetm.Solver(nx, ny, nz, wl.DXY, wl.DXY, wl.DZ, wl.DZ, "fp32", pec=pec, eps_r=eps)
    s.set_bunch(2.0 * wl.DZ, 1e-9, max(1, nx // 2), max(1, ny // 2))
    return s


def fields(s):
    return [s.get(c) for c in COMPS]


# one node; one tile and one past it in each direction; planes below, at and
# above the shortest chunk and the longest; more tiles than two per SM
@pytest.mark.parametrize("n", [(2, 2, 2), (56, 12, 4), (57, 13, 5), (64, 64, 130), (113, 25, 67), (240, 230, 9)])
@pytest.mark.parametrize("kind", ["box", "pec", "mat"])
def test_chunks_same_fields(n, kind):
    s = build(n, kind)
    info = s.info()
    assert 4 <= info["chunk_z"] <= 64
    s.step(7)
    want = fields(s)
    wake = s.wake()[0]
    s.close()
    for cz in (4, 5, 32, 200):
        s = build(n, kind)
        s.set_tiling(0, 0, cz)
        assert s.info()["chunk_z"] == cz
        s.step(7)
        for a, b in zip(want, fields(s)):
            assert np.array_equal(a, b)
        # samples are summed in float64 in any order: n additions of one rounding each
        got = s.wake()[0]
        assert np.abs(got - wake).max() <= 4 * n[2] * np.finfo(float).eps * max(np.abs(wake).max(), 1e-300)
        s.close()


@pytest.mark.parametrize("n", [(57, 13, 5), (113, 25, 67)])
def test_items_of_an_open_box(n):
    s = build(n, "box")
    cz = s.info()["chunk_z"]
    assert s.info()["work_items"] == math.ceil(n[0] / 56) * math.ceil(n[1] / 12) * math.ceil(n[2] / cz)
    s.close()


def test_batch_members_choose_their_own():
    sizes = [(57, 13, 5), (64, 64, 130), (113, 25, 67)]
    want = []
    for n in sizes:
        s = build(n, "pec")
        s.step(9)
        want.append(fields(s))
        s.close()
    members = [build(n, "pec") for n in sizes]
    members[2].set_tiling(0, 0, 6)
    before = [m.info() for m in members]
    b = tetm.Batch(members, [9] * len(members), graph_steps=4)
    b.step(9)
    b.sync()
    b.close()
    for m, w, i in zip(members, want, before):
        assert m.info()["chunk_z"] == i["chunk_z"] and m.info()["work_items"] == i["work_items"]
        for x, y in zip(w, fields(m)):
            assert np.array_equal(x, y)
        m.close()
