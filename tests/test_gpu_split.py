"""Passes that go out as two launches (FP32 strips of more than 64 rows): the
bits of one plain-load launch per step, and the first launch of every pass
announces it to the second, also when the call is replayed from a graph."""
import numpy as np
import pytest

from test_gpu_parity import BUILDERS
from test_gpu_tiles import _agree

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_10241_gb300 import build
    build.build()


def _begun(s):
    """The pass number in the lattice's device word: after both distribution buffers, the partial sums (4096 blocks of
    12 doubles) and 192 bytes of results and status."""
    at = s.state_bytes() - 16
    at = 2 * at + 4096 * 12 * 8 + 192
    return int(s.buffer[at:at + 4].view(torch.int32).item())


# two and three windows, strips of some 80 rows, the last one short; one call with single steps in it
@pytest.mark.parametrize("name,nr,nz", [("cylinder_axis", 70, 19001), ("periodic_annulus", 66, 18500),
                                        ("czochralski", 1021, 1400)])
def test_split_passes_equal_one_launch_per_step(name, nr, nz):
    _agree(BUILDERS[name](nr, nz), "fp32", (8, 5, 6))


def test_every_split_pass_announces_itself():
    from paper_1806_10241_gb300.solver import Solver
    params = BUILDERS["cylinder_axis"](70, 19001)
    stream = torch.cuda.Stream()
    s, ref = (Solver(params, storage="fp32", stream=stream) for _ in range(2))
    assert _begun(s) == 0
    s.step(8)  # passes of two steps
    stream.synchronize()
    assert _begun(s) == 4
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        s.step(4)
    for _ in range(3):
        g.replay()
        torch.cuda.synchronize()
        assert _begun(s) == 6
    # the state after the replays: the steps of the graph three times over
    ref.step(8 + 3 * 4)
    assert np.array_equal(s.get_dist(), ref.get_dist())
    assert s.diag()["status"] == 0
