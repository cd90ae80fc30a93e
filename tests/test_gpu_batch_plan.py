"""Batches whose strips would be too uneven take single steps, others passes of
several steps, with the same bits."""
import os
import sys

import numpy as np
import pytest

from paper_1806_10241_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_10241_gb300 import build
    build.build()


@pytest.mark.parametrize("storage,count,launches", [("fp16", 64, 4), ("fp16", 96, 12), ("fp16", 128, 12), ("fp32", 96, 6)])
def test_uneven_batches_take_single_steps(storage, count, launches):
    import bench
    from paper_1806_10241_gb300.batch import Batch
    from paper_1806_10241_gb300.solver import Solver
    stream = torch.cuda.Stream()
    cases = W.batched_instances(count, lo=32, hi=512)
    sols = []
    for c in cases:
        sols.append(Solver(c.params, storage=storage, stream=stream))
        sols[-1].init_fields(c.fields)
    b = Batch(sols, stream=stream)
    assert bench.count_kernels(stream, lambda: b.step(12)) == launches
    b.step(5)
    for m in (0, count // 2, count - 1):
        ref = Solver(cases[m].params, storage=storage, stream=stream)
        ref.init_fields(cases[m].fields)
        ref.step(17)
        assert sols[m].step_count == 17 and np.array_equal(sols[m].get_dist(), ref.get_dist())
    b.close()
