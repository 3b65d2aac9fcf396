"""A tuned solve steps no slower than one left to the library: where its choice is a step that no shape names, the
tuner answers with that choice, and set_tiling takes the answer on a new solve."""
import pytest

from paper_0901_1053_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tetm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_0901_1053_gb300 import tetm as t
    return t


# more than ten times, and twice, as fast as any shape
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_small_solves_keep_the_two_launches(tetm, tmp_path, precision):
    from paper_0901_1053_gb300.autotune import Autotuner
    w = wl.plain_pipe(nz=192, n=48, precision=precision)
    best = Autotuner(cache_path=str(tmp_path / "c.json")).tune(w)
    assert best == (0, 0, 0)
    s = tetm.Solver.from_workload(w)
    left = s.info()
    s.set_tiling(*best)
    assert s.info() == left
    s.set_tiling(28, 20, 32)
    assert s.info()["processed_cells"] != left["processed_cells"]
    s.close()


def test_rz_float64(tetm):
    from paper_0901_1053_gb300.autotune import tune_rz
    w = wl.cavity_chain_rz(93, 771, 0, 0, precision="fp64")
    kernel, chunk = tune_rz(w)
    assert (kernel, chunk) == ("default", 0)
    s = tetm.RzSolver(w.nr, w.nz, 0, 0, w.dr, w.dz, w.cdt, "fp64", pec=w.pec)
    left = s.info()
    s.set_kernel(kernel)
    assert s.info() == left
    s.set_tiling(16)
    with pytest.raises(ValueError):
        s.set_kernel("default")
    s.close()
