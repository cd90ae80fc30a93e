"""Lattices whose geometric sources amplify disturbances keep one order of
operations on every path: the same bits for each row fetch, alone and in a
batch, beside lattices without it."""
import numpy as np
import pytest

from test_gpu_parity import BUILDERS, random_state

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_10241_gb300 import build
    build.build()


def _params(name, nr, nz, alpha):
    p = dict(BUILDERS[name](nr, nz))
    p["alpha"] = alpha
    return p


# the diffusivity at and past the line of 3 (r0 + 1/2) where the path changes; r0 = 0 in both families
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("alpha", [1.5, 1.500001, 4.0])
@pytest.mark.parametrize("name,nr,nz", [("czochralski", 65, 7), ("cylinder_axis", 193, 40), ("periodic_cylinder", 2, 2)])
def test_every_path_gives_the_same_bits(name, nr, nz, alpha, storage):
    from paper_1806_10241_gb300.batch import Batch
    from paper_1806_10241_gb300.solver import Solver
    stream = torch.cuda.Stream()
    params = _params(name, nr, nz, alpha)
    other = BUILDERS["annulus_walls"](70, 33)
    state, state2 = random_state(params, 3), random_state(other, 4)

    def solver(p, st, launch=(0, 0, 0)):
        s = Solver(p, storage=storage, stream=stream)
        s.set_launch(*launch)
        s.set_dist(st)
        return s

    ref, ref2 = solver(params, state, (4, 1, 3)), solver(other, state2)
    ref.step(9)
    ref2.step(9)
    want, want2 = ref.get_dist(), ref2.get_dist()
    assert np.all(np.isfinite(want))
    for launch in ((0, 0, 0), (3, 2, 1), (5, 1, 2), (1, 4, 3)):
        s = solver(params, state, launch)
        s.step(4)
        s.step(5)
        assert np.array_equal(s.get_dist(), want), launch
    for launch in ((0, 0, 8, 0), (4, 1, 4, 1), (3, 2, 3, 3), (4, 2, 0, 5)):
        for mixed in (False, True):
            sols = [solver(params, state)] + ([solver(other, state2)] if mixed else [])
            b = Batch(sols, stream=stream)
            b.set_launch(*launch)
            b.step(4)
            b.step(5)
            assert np.array_equal(sols[0].get_dist(), want), (launch, mixed)
            if mixed:
                assert np.array_equal(sols[1].get_dist(), want2), launch
            b.close()
