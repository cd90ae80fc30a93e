"""lb_diagnostics_static gives the bits of lb_diagnostics on long and wide
lattices too, whose reduction grids are near the limits of its scratch."""
import numpy as np
import pytest

from test_gpu_parity import BUILDERS
from test_zz_no_alloc import FIELDS, _static_diag

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_10241_gb300 import build
    build.build()


# more than 2048 blocks of 120 columns and 32 rows each; the last two beyond nr + nz = 20000
@pytest.mark.parametrize("nr,nz,bitwise", [(508, 15953, True), (9000, 1040, True), (2500, 3300, True), (24600, 320, True),
                                           (300, 26200, False)])
def test_static_diagnostics_have_the_same_bits(nr, nz, bitwise):
    from paper_1806_10241_gb300.solver import Solver
    params = BUILDERS["annulus_walls"](nr, nz)
    x, y = np.arange(nz)[:, None] / nz, np.arange(nr)[None, :] / nr
    f = np.empty((5, nz, nr))
    f[0] = 1.0 + 0.01 * np.sin(9 * x + 5 * y)
    f[1] = 0.03 * np.sin(7 * x - 3 * y)
    f[2] = 0.02 * np.cos(4 * x + 6 * y)
    f[3] = 0.01 * np.cos(x + y)
    f[4] = 0.5 + 0.3 * np.sin(11 * x + 2 * y)
    s = Solver(params, storage="fp64")  # (FP64 sums of FP32 values are nearly exact, in any order)
    s.init_fields(f)
    s.step(2)
    want, got = s.diag(), _static_diag(s, s.step_count)
    for k in FIELDS + ("nu_side",):
        if bitwise:
            assert got[k] == want[k], k
        else:
            assert got[k] == pytest.approx(want[k], rel=1e-11, abs=1e-13), k
