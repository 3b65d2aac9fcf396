"""The check of the material arrays (finite values >= 1; one value or several), on the host for few cells and on the
device for many: the same answers on both sides of the line (65536 cells)."""
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


def make(tetm, dims, **mat):
    nx, ny, nz = dims
    return tetm.Solver(nx, ny, nz, wl.DXY, wl.DXY, wl.DZ, wl.DZ, "fp32", **mat)


@pytest.mark.parametrize("dims", [(32, 32, 64), (32, 32, 65), (57, 33, 70)])  # at the line, above it
@pytest.mark.parametrize("which", ["eps_r", "mu_r"])
def test_values(tetm, dims, which):
    nx, ny, nz = dims
    good = np.full((nz, ny, nx), 2.0)
    for at in (0, good.size // 2 + 1, good.size - 1):
        for bad in (0.999, np.nan, np.inf, -2.0):
            a = good.copy()
            a.flat[at] = bad
            with pytest.raises(Exception, match="bad argument"):
                make(tetm, dims, **{which: a})
        a = good.copy()
        a.flat[at] = 2.5
        s = make(tetm, dims, **{which: a})
        assert s.info()["tile_y"] == 12  # several materials
        s.close()
    s = make(tetm, dims, **{which: good})
    assert s.info()["tile_y"] == 28  # one
    s.close()
    # one array uniform, the other not; one wrong
    a = good.copy()
    a.flat[-1] = 3.0
    other = "mu_r" if which == "eps_r" else "eps_r"
    s = make(tetm, dims, **{which: a, other: good})
    assert s.info()["tile_y"] == 12
    s.step(2)
    s.close()
    a.flat[-1] = 0.0
    with pytest.raises(Exception, match="bad argument"):
        make(tetm, dims, **{which: a, other: good})
