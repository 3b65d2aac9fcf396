"""The autotuners' answer where the library's own choice is the fastest step, which no shape or kernel name names, and
a cache that outlived the kernels it was filled for. Host logic only: timings are stand-ins."""
import types

import numpy as np
import pytest

from paper_0901_1053_gb300 import autotune, build, tetm


def workload(precision="fp32"):
    pec = np.zeros((40, 48, 64), np.uint8)
    pec[:, :4, :] = 1
    return types.SimpleNamespace(nx=64, ny=48, nz=40, pec=pec, precision=precision)


class Timed(autotune.Autotuner):
    """Shapes take a second each, the library's choice `own` seconds."""

    def __init__(self, path, own):
        super().__init__(cache_path=str(path))
        self.own = own
        self.calls = 0

    def measure(self, w, precision, shapes, eps_r=None):
        self.calls += 1
        self.default_seconds = self.own
        return {tuple(s): 1.0 + 1e-3 * i for i, s in enumerate(shapes)}

    def wave_fitted(self, w, precision, tile_ys=(12, 20, 28), max_extra=6, eps_r=None):
        return []


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_the_librarys_choice_wins_and_is_cached(tmp_path, precision):
    t = Timed(tmp_path / "c.json", 0.5)
    assert t.tune(workload(precision)) == (0, 0, 0) == autotune.DEFAULT
    u = Timed(tmp_path / "c.json", 2.0)
    assert u.tune(workload(precision)) == (0, 0, 0) and u.calls == 0
    assert Timed(tmp_path / "d.json", 2.0).tune(workload(precision)) != (0, 0, 0)


def test_batches_and_given_candidates_get_a_shape(tmp_path):
    t = Timed(tmp_path / "c.json", 0.5)
    assert t.tune(workload(), batch=True) != (0, 0, 0)
    assert t.tune(workload("fp64"), candidates=[(28, 12, 16)]) == (28, 12, 16)


def test_measure_times_the_librarys_choice_before_any_shape(monkeypatch):
    calls = []

    class Solver:
        def __init__(self, *a, **k):
            pass

        def set_tiling(self, *shape):
            if shape[0] == 32:
                raise tetm.TetmError(tetm.TETM_E_UNSUPPORTED, "set_tiling")
            calls.append(shape)

        def step(self, n):
            calls.append(n)

        def sync(self):
            pass

        def close(self):
            calls.append("close")

    monkeypatch.setattr(tetm, "Solver", Solver)
    w = types.SimpleNamespace(nx=4, ny=4, nz=4, dx=1.0, dy=1.0, dz=1.0, cdt=1.0, pec=None)
    t = autotune.Autotuner(cache_path="/nonexistent/c.json", steps=7, warmup=2, repeats=1)
    out = t.measure(w, "fp64", [(28, 20, 32), (32, 8, 64)])
    assert list(out) == [(28, 20, 32)] and t.default_seconds > 0
    assert calls == [2, 7, (28, 20, 32), 2, 7, "close"]


def test_a_cache_filled_for_other_kernels_is_not_used(tmp_path, monkeypatch):
    src = tmp_path / "csrc"
    src.mkdir()
    (src / "k.cu").write_text("// a kernel\n")
    monkeypatch.setattr(build, "CSRC", str(src))
    t = Timed(tmp_path / "c.json", 2.0)
    first = t.tune(workload())
    assert t.tune(workload()) == first and t.calls == 1
    (src / "k.cu").write_text("// the kernel, changed\n")
    u = Timed(tmp_path / "c.json", 0.5)
    assert u.tune(workload()) == (0, 0, 0) and u.calls == 1


class Rz:
    """A solve whose kernels take 1 s a step (bulk2) or 2, and whose own choice in float64 takes `own`."""
    own = 0.5
    clock = 0.0

    def __init__(self, nr, nz, m_lo, m_hi, dr, dz, cdt, precision, pec=None):
        self.kernel, self.chunks, self.precision = None, [], precision

    def info(self):
        return {"chunk_z": 2 if self.precision == "fp32" else 8}

    def set_kernel(self, k):
        self.kernel = k

    def set_tiling(self, c):
        assert c >= 4
        self.chunk = c

    def wave_fitted_chunk(self):
        return 40

    def step(self, n):
        one = Rz.own if self.kernel is None else {"bulk2": 1.0}.get(self.kernel, 2.0) + 1e-3 * self.chunk
        Rz.clock += n * one

    def sync(self):
        pass

    def close(self):
        pass


def test_rz_tuner_knows_the_librarys_choice(monkeypatch):
    monkeypatch.setattr(tetm, "RzSolver", Rz)
    monkeypatch.setattr(autotune.time, "perf_counter", lambda: Rz.clock)
    w = types.SimpleNamespace(nr=8, nz=8, m_lo=0, m_hi=0, dr=1.0, dz=1.0, cdt=1.0, pec=None, precision="fp64")
    assert autotune.tune_rz(w) == ("default", 0)
    monkeypatch.setattr(Rz, "own", 3.0)
    assert autotune.tune_rz(w) == ("bulk2", 8)                   # the library's chunk is among those timed
    assert autotune.tune_rz(w, "fp32") == ("bulk2", 4)           # no shorter than a chunk that can be set
