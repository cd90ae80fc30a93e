"""The number of kernel launches that the benchmark reports is the number that
a call makes: passes of several steps, two launches for a split one."""
import os
import sys

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


# three and two steps per pass on resident tiles, two on strips (as one launch and as two), four, one
@pytest.mark.parametrize("nr,nz,storage,launches", [(100, 100, "fp32", 4), (256, 512, "fp32", 6), (512, 600, "fp32", 6),
                                                    (1024, 2048, "fp32", 12), (512, 1024, "fp16", 4), (41, 41, "fp64", 12)])
def test_launches_of_a_call(nr, nz, storage, launches):
    import bench
    from paper_1806_10241_gb300.solver import Solver
    c = W.swirling_cylinder(nr=nr, nz=nz, Re=200.0, Ra=1e4)
    s = Solver(c.params, storage=storage, stream=torch.cuda.Stream())
    assert bench.count_kernels(s.stream, lambda: s.step(12)) == launches
    assert s.step_count == 12 and s.diag()["status"] == 0


def test_launches_of_a_batch():
    import bench
    from paper_1806_10241_gb300.batch import Batch
    from paper_1806_10241_gb300.solver import Solver
    stream = torch.cuda.Stream()
    sols = [Solver(c.params, storage="fp32", stream=stream) for c in W.batched_instances(6, lo=32, hi=96)]
    b = Batch(sols, stream=stream, graph_steps=4)
    assert bench.count_kernels(stream, lambda: b.step(12)) < 12
    b.set_launch(seg_rows=8, graph_steps=0)
    assert bench.count_kernels(stream, lambda: b.step(9)) == 9
    assert all(s.step_count == 21 for s in sols) and all(d["status"] == 0 for d in b.diag())
    b.close()
