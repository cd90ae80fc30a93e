"""Lattices past the line from which the arithmetic keeps one order of
operations (max(nu, alpha) > 3 (r0 + 1/2)) against the oracle, alone and in a
batch, and the row fetch that they report."""
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


def _stepped(params, state, n):
    o = oracle.Oracle(params)
    o.set_dist(state)
    o.step(n)
    return o.get_dist()


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("more", [{"alpha": 1.6}, {"alpha": 4.0}, {"nu": 2.0}, {"alpha": 2.5, "explicit_sources": 1}])
@pytest.mark.parametrize("name,nr,nz", [("cylinder_axis", 2, 5), ("czochralski", 65, 9), ("periodic_cylinder", 193, 17),
                                        ("rotating_cylinder", 65, 12)])
def test_distributions_match_the_oracle(name, nr, nz, more, storage):
    from paper_1806_10241_gb300.batch import Batch
    from paper_1806_10241_gb300.solver import Solver
    params = dict(BUILDERS[name](nr, nz), **more)
    stream = torch.cuda.Stream()
    rest = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4 + [0] * 5 + [0] * 5)[:, None, None] * params["rho0"] + \
        np.array([0] * 14 + [1 / 3] + [1 / 6] * 4)[:, None, None] * params["T0"]
    steps = 3 if storage == "fp32" else 1
    for batched in (False, True):
        s = Solver(params, storage=storage, stream=stream)
        s.set_dist(random_state(params, 23))
        state = s.get_dist()  # as stored
        want = _stepped(params, state, steps)
        # how the lattice itself amplifies a disturbance over these steps
        eps = 1e-9
        noise = np.random.default_rng(1).choice([-1.0, 1.0], state.shape)
        grown = np.max(np.abs(_stepped(params, state + eps * noise, steps) - want)) / eps
        if storage == "fp16":  # deviations times 2^10 saturate at the largest FP16 number
            want = rest + np.clip(want - rest, -65504 / 1024, 65504 / 1024)
        if batched:
            b = Batch([s], stream=stream)
            b.step(steps)
            b.close()
        else:
            s.step(steps)
        # FP32: 2e-6 as in the parity tests (round-off times the operations that touch a value), as far as it grows; 16
        # bits: one rounding to a neighbour, 2^-10 or 2^-7 of the deviation from rest (FP16 subnormals: 2^-34) besides
        tol = 2e-6 * max(1.0, grown)
        if storage != "fp32":
            tol = tol + np.abs(want - rest) * (2.0 ** -10 if storage == "fp16" else 2.0 ** -7)
        assert np.all(np.abs(s.get_dist() - want) <= tol), (batched, np.max(np.abs(s.get_dist() - want) - tol))


def test_pinned_lattices_report_their_row_fetch():
    from paper_1806_10241_gb300.solver import Solver
    for alpha, fetch in ((1.5, 1), (1.6, 3)):
        s = Solver(dict(BUILDERS["cylinder_axis"](40, 12), alpha=alpha), storage="fp32")
        s.set_launch(5, 2, 1)
        assert s.get_launch() == (5, 2, fetch)
    s = Solver(dict(BUILDERS["cylinder_axis"](40, 12), alpha=1.6), storage="fp64")
    assert s.get_launch()[2] == 1
