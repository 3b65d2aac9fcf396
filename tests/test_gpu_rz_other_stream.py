"""A rotationally symmetric solve stepped on a stream of the caller's right after its creation, which works on a
stream of the library's own: everything the step kernels read is there when tetm_rz_create returns. Grids of two
planes take the shortest way through the choice of the chunk length; their fields are the same bits on either stream
(the same operations in the same order)."""
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


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nr,nz", [(8, 2), (700, 2), (57, 3), (130, 90)])
def test_first_step_on_another_stream(tetm, nr, nz, precision):
    pec = wl.cavity_chain_rz(nr, nz, 0, 1).pec
    pec[-1, nr // 2:] = 1          # the activity changes from plane to plane
    side = torch.cuda.Stream()
    rng = np.random.default_rng(nr)
    start = rng.standard_normal((2, 6, nz + 1, nr + 1))
    got = []
    for stream in (0, side.cuda_stream):
        s = tetm.RzSolver(nr, nz, 0, 1, 1e-3, 1e-3, 1e-3, precision, pec=pec)
        s.set_stream(stream)
        for m in (0, 1):
            for c in range(6):
                s.set(m, c, start[m, c])
        s.step(5)
        got.append([s.get(m, c) for m in (0, 1) for c in range(6)])
        s.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
