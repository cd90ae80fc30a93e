"""The FP64 step on blocks of rows of a 32-column window: every boundary
family at the edges of windows and blocks against the oracle, and the same
bits for every number of rows and warps per block (one and two warps per row
differ in which planes a warp stores, not in its arithmetic)."""
import numpy as np
import pytest

import oracle
from test_gpu_parity import BUILDERS, random_state

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_10241_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("nr,nz", [(2, 2), (31, 5), (32, 3), (33, 7), (64, 17), (65, 40)])
@pytest.mark.parametrize("name", list(BUILDERS))
def test_fp64_step_matches_oracle_for_every_block_shape(name, nr, nz):
    from paper_1806_10241_gb300.solver import Solver
    params = BUILDERS[name](nr, nz)
    state = random_state(params, 11)
    ref = oracle.Oracle(params)
    ref.set_dist(state)
    ref.step(3)
    first = None
    for launch in ((0, 0, 0), (1, 1, 1), (2, 4, 1), (3, 8, 1), (16, 2, 1), (40, 5, 1), (32, 8, 3)):
        s = Solver(params, storage="fp64")
        s.set_launch(*launch)
        s.set_dist(state)
        s.step(3)
        got = s.get_dist()
        s.close()
        # 1e-12: the bar of the FP64 parity tests (a few hundred operations of round-off 1e-16 on values below 1)
        assert np.max(np.abs(got - ref.get_dist())) < 1e-12, (name, launch)
        if first is None:
            first = got
        assert np.array_equal(got, first), (name, launch)
