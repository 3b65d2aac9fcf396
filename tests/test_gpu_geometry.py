"""Which entries carry a field, from the cells around them, with one material (mask only) and with material arrays.
Whole numbers: no tolerance."""
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


def expected(pec):
    """Entry (c, k, j, i) is active where every cell around the edge or face is open (cells outside are closed)."""
    nz, ny, nx = pec.shape
    o = np.zeros((nz + 2, ny + 2, nx + 2), bool)
    o[1:-1, 1:-1, 1:-1] = pec == 0

    def at(di, dj, dk):
        return o[1 + dk:nz + 2 + dk, 1 + dj:ny + 2 + dj, 1 + di:nx + 2 + di]

    own, x, y, z = at(0, 0, 0), at(-1, 0, 0), at(0, -1, 0), at(0, 0, -1)
    return [own & y & z & at(0, -1, -1), own & x & z & at(-1, 0, -1), own & x & y & at(-1, -1, 0), own & x, own & y, own & z]


@pytest.mark.parametrize("dims", [(2, 2, 2), (15, 15, 3), (16, 16, 5), (33, 7, 70)])  # nodes of a plane below, at, above a block
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
@pytest.mark.parametrize("kind", ["vacuum", "eps", "mu"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_active_entries(tetm, dims, share, kind, precision):
    nx, ny, nz = dims
    rs = np.random.default_rng(11)
    pec = (rs.uniform(size=(nz, ny, nx)) < share).astype(np.uint8)
    m = np.where(rs.uniform(size=pec.shape) < 0.5, 1.0, 2.5)
    m[0, 0, 0], m[-1, -1, -1] = 1.0, 2.5
    s = tetm.Solver(nx, ny, nz, wl.DXY, wl.DXY, wl.DZ, wl.DZ, precision, pec=pec,
                    eps_r=m if kind == "eps" else None, mu_r=m if kind == "mu" else None)
    want = expected(pec)
    assert s.info()["active_cells"] == int(np.logical_or.reduce(want).sum())
    for c, w in enumerate(want):
        s.set(c, np.ones(s.shape))
        got = np.asarray(s.get(c)).reshape(nz + 1, ny + 1, nx + 1)
        assert np.array_equal(got != 0, w)
    s.close()
