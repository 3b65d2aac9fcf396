"""The float64 default step (two launches over bands of rows of every plane) against the warp-tiled sweep, which
the parity tests hold to the oracle.

Tolerance: none. Both do the same operations per node in the same order, so fields and wakes are the same bits; the
energy sums the same terms in another grouping, within 1e-12 of its value."""
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


def run(tetm, dims, tiling, pec, eps=None, mu=None):
    nx, ny, nz = dims
    s = tetm.Solver(nx, ny, nz, wl.DXY, wl.DXY, wl.DZ, wl.DZ, "fp64", pec=pec, eps_r=eps, mu_r=mu)
    if tiling:
        s.set_tiling(*tiling)
    s.set_bunch(2.3 * wl.DZ, 1e-9, nx // 2, ny // 2)
    s.set_observer(nx // 2 - 1, ny // 2 - 1)
    for c, a in enumerate(wl.random_fields(s.shape, 5)):
        s.set(c, a)
    s.step(7)
    out = [s.get(c) for c in range(6)] + [s.wake()[0], *s.transverse_wake()]
    e = s.energy()
    assert s.check_guards() == 0
    s.close()
    return out, e


# band edges: fewer rows than a band, whole bands, a remainder; column cuts at 64: one item, two, three; the last
# grid has enough cells for the longer bands
@pytest.mark.parametrize("dims", [(2, 2, 2), (3, 8, 5), (64, 9, 6), (65, 17, 9), (130, 16, 4), (129, 70, 130)])
@pytest.mark.parametrize("geometry", ["box", "random", "materials"])
def test_band_step_is_bitwise_the_warp_sweep(tetm, dims, geometry):
    nx, ny, nz = dims
    pec = eps = mu = None
    if geometry == "random":   # holes, empty bands and detached columns
        rng = np.random.default_rng(sum(dims))
        pec = (rng.uniform(size=(nz, ny, nx)) < 0.2).astype(np.uint8)
        pec[:, : ny // 3] = 1
        pec[nz // 2] = 1
    elif geometry == "materials":
        eps, mu, pec = wl.random_materials(nx, ny, nz, 3)
    (a, ea), (b, eb) = (run(tetm, dims, t, pec, eps, mu) for t in (None, (28, 12, 8)))
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    assert abs(ea - eb) <= 1e-12 * max(abs(eb), 1e-300)
