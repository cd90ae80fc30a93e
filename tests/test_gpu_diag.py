"""Fields and diagnostics on blocks of 128 columns and 4 to 32 rows: every
boundary family at the edges of those blocks against the oracle, and fields
moved in several pieces."""
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


# one block short of, at and past its 128 columns and 4 rows; a lattice whose blocks have 32 rows; one cut into pieces
@pytest.mark.parametrize("storage", ["fp64", "fp32", "bf16", "fp16"])
@pytest.mark.parametrize("nr,nz", [(2, 2), (3, 3), (127, 4), (128, 5), (129, 9), (257, 8), (129, 4865)])
@pytest.mark.parametrize("name", list(BUILDERS))
def test_fields_and_diagnostics_match_oracle_at_block_edges(name, nr, nz, storage):
    from paper_1806_10241_gb300.solver import Solver
    params = BUILDERS[name](nr, nz)
    s = Solver(params, storage=storage)
    s.set_dist(random_state(params, 5))
    s.step(1)
    o = oracle.Oracle(params)
    o.set_dist(s.get_dist())
    got, want, dg, do = s.fields(), o.fields(), s.diag(), o.diag()
    # FP64: the bars of the parity tests.  Else FP32 arithmetic on the stored values: sums of at most 9 terms below 1
    # and one division, 16 roundings of 2^-24 on values below 2
    tol = 1e-12 if storage == "fp64" else 2e-6
    assert np.max(np.abs(got - want)) < tol
    assert dg["T_sum"] == pytest.approx(do["T_sum"], rel=tol, abs=tol)
    assert dg["u_max"] == pytest.approx(do["u_max"], abs=tol)
    assert dg["mass"] == pytest.approx(do["mass"], rel=1e-11, abs=tol * nr * nz)
    # a wall gradient of the temperature over a length of the lattice: weights (8 + 9 + 1) / 3
    for k in range(4):
        assert dg["nu_side"][k] == pytest.approx(do["nu_side"][k], rel=1e-11, abs=6 * tol * max(nr, nz)), k


@pytest.mark.parametrize("storage", ["fp64", "fp16"])
@pytest.mark.parametrize("nr,nz", [(1023, 103), (70, 1501), (2050, 1500)])
def test_fields_moved_in_pieces_round_trip(nr, nz, storage):
    """Exchanges above and below the size from which copies and kernels
    overlap: the fields that were set are those of the state, and pageable and
    pinned memory receive the same values, on a stream of the caller's."""
    from paper_1806_10241_gb300.solver import Solver
    params = BUILDERS["periodic_cylinder"](nr, nz)
    f = np.zeros((5, nz, nr))
    f[0] = 1.0
    f[4] = np.arange(nz)[:, None] % 17 * 0.05 + np.arange(nr) % 5 * 0.01  # each piece has its own rows
    s = Solver(params, storage=storage, stream=torch.cuda.Stream())
    s.init_fields(f)
    # FP64: round-off; FP16: the five parts of T, each with deviations below 1/2 held to 11 bits
    assert np.max(np.abs(s.get_dist()[14:].sum(axis=0) - f[4])) < (1e-13 if storage == "fp64" else 2e-3)
    a = s.fields()
    pinned = torch.empty(5, nz, nr, dtype=torch.float64, pin_memory=True).numpy()
    assert np.array_equal(s.fields(out=pinned), a)
    assert s.diag()["T_sum"] == pytest.approx(a[4].sum(), rel=1e-6)
