"""Lattices and batches let go of while their launches are queued: their
device memory is not handed out again before these are done."""
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


def _range(t):
    return t.data_ptr(), t.data_ptr() + t.numel()


def _apart(new, old):
    a, b = _range(new)
    return b <= old[0] or old[1] <= a


def _solver(stream):
    from paper_1806_10241_gb300.solver import Solver
    c = W.swirling_cylinder(nr=256, nz=512, Re=200.0, Ra=1e4)
    s = Solver(c.params, storage="fp16", stream=stream)
    s.init_fields(c.fields)
    return s


def _while_busy(attempt):
    """attempt() -> (whether its work was still queued, whether its memory was apart), until the first holds."""
    for _ in range(5):
        busy, apart = attempt()
        torch.cuda.synchronize()
        if busy:
            return apart
    pytest.skip("the work was done too soon")


def test_lattice_dropped_with_work_queued():
    def attempt():
        stream = torch.cuda.Stream()
        s = _solver(stream)
        s.step(20000)  # some ten milliseconds are still queued on return
        old, n = _range(s.buffer), s.buffer.numel()
        del s
        again = torch.empty(n, dtype=torch.uint8, device="cuda")
        return not stream.query(), _apart(again, old)

    assert _while_busy(attempt)


def test_batch_dropped_with_work_queued():
    from paper_1806_10241_gb300.batch import Batch

    def attempt():
        stream = torch.cuda.Stream()
        sols = [_solver(torch.cuda.current_stream()) for _ in range(2)]
        b = Batch(sols, stream=stream)
        b.step(20000)
        buffers = [b.buffer] + [s.buffer for s in sols]
        old, sizes = [_range(t) for t in buffers], [t.numel() for t in buffers]
        del b, sols, buffers
        again = [torch.empty(n, dtype=torch.uint8, device="cuda") for n in sizes]
        return not stream.query(), all(_apart(t, o) for t in again for o in old)

    assert _while_busy(attempt)
