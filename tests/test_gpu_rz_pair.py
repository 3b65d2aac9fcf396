"""The float32 two-step sweep with packed arithmetic, alone (kernel bulk2) and as the default's pairs of steps, against
the register-ring sweep, which the parity tests hold to the oracle.

Tolerance: none. Both round every operation alike and in the same order, so fields and wakes are the same bits."""
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


def run(tetm, kernel, chunk, nr, nz, modes, pec, start="cold", fields=True, steps=9, eps=None):
    s = tetm.RzSolver(nr, nz, modes[0], modes[-1], 1e-3, 1e-3, 1e-3, "fp32", pec=pec, eps_r=eps)
    if kernel:
        s.set_kernel(kernel)
    if chunk:
        s.set_tiling(chunk)
    if start == "cold":
        s.set_bunch(2.2e-3, 1e-9, 0 if modes == (0,) else 2)
    else:
        s.set_bunch_scattered(2.2e-3, 1e-9, 2, 28)
    rng = np.random.default_rng(3)
    for m in modes if fields else ():
        for c in range(6):
            s.set(m, c, rng.standard_normal(s.shape))
    for n in (steps - 3, 2, 1):   # pairs with an odd rest, a call of two, a call of one
        s.step(n)
    out = [x for m in modes for x in [s.get(m, c) for c in range(6)] + [s.wake(m)[0], s.transverse_wake(m)]]
    assert s.check_guards() == 0
    s.close()
    return out


def same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


# one window and several (56 owned entries), items of few planes down to one, longer than the grid; 33 planes: items
# cross a word of change bits
@pytest.mark.parametrize("nr,nz", [(8, 2), (9, 5), (56, 33), (57, 70), (130, 90), (300, 33)])
@pytest.mark.parametrize("kernel,chunk", [(None, None), ("bulk2", None), ("bulk2", 4), ("bulk2", 5), ("bulk2", 100)])
@pytest.mark.parametrize("geometry", ["chain", "random"])
def test_pair_sweep_is_bitwise_the_register_sweep(tetm, nr, nz, kernel, chunk, geometry):
    pec = wl.cavity_chain_rz(nr, nz, 0, 2).pec
    if geometry == "random":   # the activity changes at every plane
        pec = (np.random.default_rng(nr + nz).uniform(size=(nz, nr)) < 0.1).astype(np.uint8)
        pec[:, :3] = 0
    same(run(tetm, kernel, chunk, nr, nz, (0, 1, 2), pec), run(tetm, "register", 16, nr, nz, (0, 1, 2), pec))


@pytest.mark.parametrize("modes,start,steps", [((0,), "cold", 60), ((1, 2), "cold", 61), ((0, 1), "scattered", 160)])
def test_pair_sweep_with_the_bunch_alone(tetm, modes, start, steps):
    pec = wl.cavity_chain_rz(64, 512, 0, 2).pec
    a = run(tetm, None, None, 64, 512, modes, pec, start, False, steps)
    same(a, run(tetm, "register", 16, 64, 512, modes, pec, start, False, steps))
    same(a, run(tetm, "bulk2", 7, 64, 512, modes, pec, start, False, steps))


def test_default_keeps_the_state_before_the_last_step(tetm):
    """The default takes pairs of steps but ends a call on a single one: the charges stay available."""
    w = wl.cavity_chain_rz(64, 512, 0, 1)
    s = tetm.RzSolver(w.nr, w.nz, 0, 1, w.dr, w.dz, w.cdt, "fp32", pec=w.pec)
    s.set_bunch(w.sigma, w.charge, w.i0)
    s.step(40)
    e, h, q = s.charge_residual(1)
    assert q > 0 and e <= 1e-3 * q
    s.close()


def test_default_chunk_with_material_arrays(tetm):
    """Material arrays stay on the register sweep, whose items the default length cuts anew."""
    rng = np.random.default_rng(5)
    eps, pec = rng.uniform(1, 4, (70, 57)), wl.cavity_chain_rz(57, 70, 0, 1).pec
    same(run(tetm, None, None, 57, 70, (0, 1), pec, eps=eps), run(tetm, "register", 16, 57, 70, (0, 1), pec, eps=eps))
