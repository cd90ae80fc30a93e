"""Several steps per launch on tiles in shared memory (the automatic launch):
the bits of one plain-load launch per step, for every boundary family, at the
edges of the windows, tiles and strips, and for every number of steps that a
call can be cut into."""
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


def _agree(params, storage, calls, seed=7):
    from paper_1806_10241_gb300.solver import Solver
    state = random_state(params, seed)
    plain, tiled = Solver(params, storage=storage), Solver(params, storage=storage)
    plain.set_launch(4, 1, 1)
    for s in (plain, tiled):
        s.set_dist(state)
    for n in calls:
        plain.step(n)
        tiled.step(n)
        assert tiled.step_count == plain.step_count
        assert tiled.diag()["status"] in (0, 4) and tiled.diag() == plain.diag()
        assert np.array_equal(tiled.get_dist(), plain.get_dist()), (params["nr"], params["nz"], n)
    # the current buffer alternates with the step count on both paths: the caller's buffer holds the same state
    half = tiled.state_bytes() - 16
    a, b = ([s.buffer[i * half:(i + 1) * half] for i in (0, 1)] for s in (plain, tiled))
    cur = sum(calls) & 1
    assert plain.get_state()[16:] == a[cur].cpu().numpy().tobytes()
    assert tiled.get_state()[16:] == b[cur].cpu().numpy().tobytes()


# widths around one and two windows (64 columns, margins of 2 and 4), heights around one and two tiles
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nr,nz", [(2, 2), (7, 3), (64, 5), (65, 9), (121, 12), (124, 13), (125, 14), (181, 47)])
@pytest.mark.parametrize("name", list(BUILDERS))
def test_tiles_equal_one_launch_per_step(name, nr, nz, storage):
    _agree(BUILDERS[name](nr, nz), storage, (1, 2, 3, 4, 5, 7, 12))


# lattices too large for resident tiles: one and more waves of strips, the last strip short
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("name,nr,nz", [("cylinder_axis", 521, 700), ("czochralski", 1023, 610), ("annulus_walls", 70, 9001),
                                        ("periodic_annulus", 66, 9001), ("free_ends_annulus", 1283, 517)])
def test_strips_equal_one_launch_per_step(name, nr, nz, storage):
    _agree(BUILDERS[name](nr, nz), storage, (1, 5, 8))


# a batch on resident tiles, and one too large for them, uneven lattices with a periodic and a split-top one among them
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("shapes", [[("cylinder_axis", 33, 17), ("periodic_annulus", 66, 12), ("czochralski", 125, 31),
                                     ("planar_box", 2, 2)],
                                    [("cylinder_axis", 513, 301), ("periodic_annulus", 70, 1500), ("czochralski", 640, 333),
                                     ("annulus_walls", 65, 4000), ("free_ends_annulus", 20, 9), ("sliding_annulus", 700, 411)]])
def test_batched_tiles_equal_one_launch_per_step(shapes, storage):
    from paper_1806_10241_gb300.batch import Batch
    from paper_1806_10241_gb300.solver import Solver
    stream = torch.cuda.Stream()
    params = [BUILDERS[name](nr, nz) for name, nr, nz in shapes]
    plain, tiled = ([Solver(p, storage=storage, stream=stream) for p in params] for _ in range(2))
    for seed, (a, b, p) in enumerate(zip(plain, tiled, params)):
        a.set_launch(4, 1, 1)
        state = random_state(p, seed)
        a.set_dist(state)
        b.set_dist(state)
    batch = Batch(tiled, stream=stream, graph_steps=4)
    for n in (1, 2, 5, 7, 8):
        batch.step(n)
        for (name, nr, nz), a, b in zip(shapes, plain, tiled):
            a.step(n)
            assert b.step_count == a.step_count
            assert np.array_equal(a.get_dist(), b.get_dist()), (name, nr, nz, n)
    batch.close()
