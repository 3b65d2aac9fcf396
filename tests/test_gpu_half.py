"""The float32 step of a small grid in two launches (runs of planes, 56 x 14 nodes) against the block-tiled sweep,
which the parity tests hold to the oracle.

Tolerance: none for the fields, both do the same operations per node in the same order. A wake sample is a float64
sum of the same terms in any order: n additions of one rounding each."""
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


def run(tetm, dims, pec, line, observer, sweep, steps=7):
    nx, ny, nz = dims
    s = tetm.Solver(nx, ny, nz, wl.DXY, wl.DXY, wl.DZ, wl.DZ, "fp32", pec=pec)
    if sweep:
        s.set_tiling(0, 0, 5)
    s.set_bunch(2.3 * wl.DZ, 1e-9, *line)
    s.set_observer(*observer)
    for c, a in enumerate(wl.random_fields(s.shape, 5)):
        s.set(c, a)
    s.step(steps)
    out = [s.get(c) for c in range(6)]
    wakes = [s.wake()[0], *s.transverse_wake()]
    assert s.check_guards() == 0
    s.close()
    return out, wakes


# tile edges: one cell, one tile, one past it in each direction; runs of one plane (few tiles), of two and more, with
# a short last run
@pytest.mark.parametrize("dims", [(2, 2, 2), (3, 40, 9), (56, 14, 8), (57, 15, 9), (24, 24, 96), (113, 43, 19),
                                  (64, 64, 131), (120, 60, 127)])
@pytest.mark.parametrize("walls", [False, True])
def test_same_as_the_sweep(tetm, dims, walls):
    nx, ny, nz = dims
    pec = (np.random.default_rng(3).uniform(size=(nz, ny, nx)) < 0.2).astype(np.uint8) if walls else None
    # the lines at the last column and row a tile owns and at the first of the next one, where the grid has them
    line = (min(55, nx - 1), min(13, ny - 1))
    observer = (min(56, nx - 1), min(14, ny - 1))
    (a, wa), (b, wb) = run(tetm, dims, pec, line, observer, False), run(tetm, dims, pec, line, observer, True)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    for x, y in zip(wa, wb):
        assert np.abs(x - y).max() <= 4 * nz * np.finfo(float).eps * max(np.abs(y).max(), 1e-300)
