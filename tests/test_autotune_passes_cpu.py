"""What the autotuner times and how it keeps it: candidates in calls of whole
passes, launches of pinned lattices apart from the others', and none from other
kernels."""
import json
import os

import pytest

from paper_1806_10241_gb300 import autotune, build, serving
from test_autotune_cpu import FakeBatch, FakeSolver


class Solver(FakeSolver):
    def __init__(self, storage="fp32", alpha=0.05, nr=64, nz=64, **more):
        super().__init__(storage, nr, nz)
        self.params = {"nr": nr, "nz": nz, "nu": 0.05, "alpha": alpha, **more}
        self.stream, self.calls = None, []

    def step(self, n=1):
        self.calls.append(n)

    def get_launch(self):
        return (4, 1, 3)


class Batch(FakeBatch):
    def __init__(self, solvers):
        super().__init__(resident=1000, items=50)
        self.solvers, self.calls = solvers, []

    def step(self, n=1):
        self.calls.append(n)


@pytest.fixture
def cache(tmp_path, monkeypatch):
    path = tmp_path / "autotune.json"
    monkeypatch.setattr(autotune, "_CACHE", str(path))
    monkeypatch.setattr(autotune, "_time", lambda stream, fn, steps: fn(steps) or 1.0)
    return path


def passes(n, T):
    """The passes of a call, as lb_step cuts it."""
    m = -(-n // T)
    m += (n - m) & 1
    return [n // m + (p < n % m) for p in range(m)]


@pytest.mark.parametrize("steps", [1, 3, 20, 24, 30])
def test_candidates_are_timed_over_whole_passes(cache, steps):
    solver, batch = Solver(), Batch([Solver()])
    autotune.tune_solver(solver, steps=steps)
    autotune.tune_batch(batch, steps=steps)
    for calls, candidates in ((solver.calls, 1 + len(autotune.SOLVER_CANDIDATES)), (batch.calls, len(batch.calls) // 2)):
        assert len(calls) == 2 * candidates > 2  # a warm-up and a timed call each
        for warm, timed in zip(calls[::2], calls[1::2]):
            for T in (2, 3, 4):
                assert timed >= steps and set(passes(timed, T)) == {T}
                assert min(passes(warm, T)) >= 2  # not the kernel of single steps


def test_server_asks_for_whole_passes():
    assert serving.WHOLE_PASSES == autotune.WHOLE_PASSES


def test_pinned_lattices_have_entries_of_their_own(cache):
    plain, pinned = Solver(), Solver(alpha=4.0)
    assert not autotune._pinned(plain) and autotune._pinned(pinned)
    assert not autotune._pinned(Solver("fp64", alpha=4.0)) and not autotune._pinned(Solver(alpha=4.0, planar=1))
    assert not autotune._pinned(Solver(alpha=1.5)) and autotune._pinned(Solver(alpha=1.500001))  # 3 (r0 + 1/2)
    assert not autotune._pinned(Solver(alpha=4.0, r0=10.0))
    autotune.tune_solver(pinned)
    autotune.tune_solver(plain)
    assert plain.calls  # not taken from the pinned one's entry
    keys = {autotune._batch_key(Batch([Solver(alpha=a) for a in alphas])) for alphas in
            ((0.1, 0.1, 0.1, 0.1), (4.0, 0.1, 0.1, 0.1), (4.0, 4.0, 4.0, 4.0))}
    assert len(keys) == 3 and len(json.loads(cache.read_text())) == 2


def test_cache_is_one_file_per_version_of_the_kernels(monkeypatch):
    assert build.source_hash() in os.path.basename(autotune._CACHE)
    before = build.source_hash()
    monkeypatch.setattr(build, "FLAGS", build.FLAGS + ["-DOTHER"])
    assert build.source_hash() != before
