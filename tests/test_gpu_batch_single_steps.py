"""Single steps of a batch under the automatic launch: work items of equal
length over all lattices, in whole waves, and the bits of every other launch."""
import numpy as np
import pytest

from paper_1806_10241_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_10241_gb300 import build
    build.build()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("kind,count,waves", [("requests", 40, 1), ("annuli", 64, 3), ("annuli", 96, 5)])
def test_single_steps_fill_whole_waves(kind, count, waves, storage):
    from paper_1806_10241_gb300.autotune import segment_plan
    from paper_1806_10241_gb300.batch import Batch
    from paper_1806_10241_gb300.solver import Solver
    cases = W.batched_instances(count, lo=32, hi=512) if kind == "annuli" else \
        [r.case for r in W.serving_requests(count=count, nr_lo=64, nr_hi=128)]
    stream = torch.cuda.Stream()
    sets = []
    for _ in range(2):
        sets.append([Solver(c.params, storage=storage, stream=stream) for c in cases])
        for s, c in zip(sets[-1], cases):
            s.init_fields(c.fields)
    auto, plain = (Batch(s, stream=stream, graph_steps=0) for s in sets)
    _, items = auto.occupancy()
    plain.set_launch(row_fetch=4 if storage == "fp32" else 3)
    resident, _ = plain.occupancy()
    shapes = [(s.nr, s.nz) for s in sets[0]]
    plan = segment_plan(shapes, resident, waves)
    assert items == sum(-(-nr // 64) * -(-nz // seg) for (nr, nz), seg in zip(shapes, plan))
    assert 0.8 * waves * resident <= items <= 1.25 * waves * resident
    plain.set_launch(seg_rows=3, warps_per_block=2, graph_steps=0, row_fetch=1)
    for n in (1, 2, 3, 1):
        auto.step(n)
        plain.step(n)
    for a, p in zip(*sets):
        assert a.step_count == p.step_count and np.array_equal(a.get_dist(), p.get_dist())
    auto.close()
    plain.close()
