"""The float64 default step of the rotationally symmetric scheme (two launches over runs of planes) against the
register-ring sweep, which the parity tests hold to the oracle.

Tolerance: none. Both do the same operations per entry in the same order, so fields and wakes are the same bits."""
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


def run(tetm, kernel, nr, nz, modes, pec, start, eps=None, mu=None, fields=(), steps=11):
    s = tetm.RzSolver(nr, nz, modes[0], modes[-1], 1e-3, 1e-3, 1e-3, "fp64", pec=pec, eps_r=eps, mu_r=mu)
    if kernel:
        s.set_kernel(kernel)
    if start == "static":
        s.set_bunch_static(2.2e-3, 1e-9, 2, 28)
    else:
        s.set_bunch(2.2e-3, 1e-9, 0 if modes == (0,) else 2)
    rng = np.random.default_rng(3)
    for m in modes:
        for c in fields:
            s.set(m, c, rng.standard_normal(s.shape))
    s.step(steps)
    out = [x for m in modes for x in [s.get(m, c) for c in range(6)] + [s.wake(m)[0], s.transverse_wake(m)]]
    assert s.check_guards() == 0
    s.close()
    return out


def same(tetm, *a, **k):
    for x, y in zip(run(tetm, None, *a, **k), run(tetm, "register", *a, **k)):
        assert np.array_equal(x, y)


# a few columns; one, two and three column cuts (256 columns); more planes than a run takes, a last short one
@pytest.mark.parametrize("nr,nz", [(4, 3), (33, 70), (255, 9), (257, 33), (530, 17)])
@pytest.mark.parametrize("geometry", ["chain", "random", "materials"])
def test_rz_band_step_is_bitwise_the_register_sweep(tetm, nr, nz, geometry):
    rng = np.random.default_rng(nr + nz)
    pec = wl.cavity_chain_rz(nr, nz, 0, 2).pec
    eps = mu = None
    if geometry != "chain":   # detached columns, empty planes
        pec = (rng.uniform(size=(nz, nr)) < 0.1).astype(np.uint8)
        pec[:, :3] = 0
        pec[nz // 2] = 1
    if geometry == "materials":
        eps, mu = rng.uniform(1, 4, (nz, nr)), rng.uniform(1, 2, (nz, nr))
    same(tetm, nr, nz, (0, 1, 2), pec, "cold", eps, mu, fields=range(6))


@pytest.mark.parametrize("modes", [(0,), (0, 1)])
@pytest.mark.parametrize("start,fields", [("cold", ()), ("static", ()), ("cold", (0, 2, 4)), ("cold", (1,)),
                                          ("cold", (3,)), ("cold", (5,))])
def test_mode_0_without_and_with_its_second_family(tetm, modes, start, fields):
    """(e_phi, h_r, h_z) of mode 0 are left out while they are zero, and taken once one of them was set."""
    if start == "static" and modes == (0,):
        modes = (0, 1, 2)
    w = wl.cavity_chain_rz(40, 512, 0, 2)
    same(tetm, 40, 512, modes, w.pec, start, fields=fields, steps=60)
