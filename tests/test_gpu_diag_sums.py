"""The sums and the largest velocity of the diagnostics are those of FP64
accumulation over the device's own node values, for every storage, also where
a lattice has overflowed."""
import math

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


def _densities(s, storage):
    """rho - rho0 of the stored state as the device forms it, [nz, nr]: FP32 sums of the stored deviations in order, FP16
    ones in storage units of 2^-10."""
    dtype = {"fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}[storage]
    raw = torch.frombuffer(bytearray(s.get_state()[16:]), dtype=dtype).to(torch.float32).numpy()
    m = 32 if storage == "fp32" else 64
    v = raw[: 19 * s.nz * (-(-s.nr // m) * m)].reshape(19, s.nz, -1)[:, :, : s.nr]
    r = v[0].copy()
    for q in range(1, 9):
        r += v[q]
    return (r * np.float32(2.0 ** -10 if storage == "fp16" else 1.0)).astype(np.float64)


# few threads with as many nodes as a thread gets, and larger lattices
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("name,nr,nz", [("cylinder_axis", 2, 64), ("annulus_walls", 3, 640), ("czochralski", 130, 96),
                                        ("periodic_annulus", 257, 1200)])
def test_sums_are_those_of_fp64(name, nr, nz, storage):
    from paper_1806_10241_gb300.solver import Solver
    params = BUILDERS[name](nr, nz)
    s = Solver(params, storage=storage)
    s.set_dist(random_state(params, 17))
    s.step(2)
    d, f, rho = s.diag(), s.fields(), _densities(s, storage)
    y = float(params.get("r0", 0.0)) + np.arange(nr) + 0.5
    # FP64 sums over a thread's, a block's and a lattice's values in turn: some dozens of roundings of 2^-53 at most, on
    # partial sums below the sum of the absolute values; FP32 pairs (2^-47) and plain FP32 sums (2^-24) fail
    eps = 2.0 ** -51
    T = f[4]
    assert abs(d["T_sum"] - math.fsum(T.ravel())) <= eps * np.abs(T).sum()
    N, sum_y = nr * nz * float(params.get("rho0", 1.0)), nz * y.sum() * float(params.get("rho0", 1.0))
    assert abs(d["mass"] - math.fsum([N] + list(rho.ravel()))) <= eps * (N + np.abs(rho).sum())
    assert abs(d["mass_r"] - math.fsum([sum_y] + list((rho * y).ravel()))) <= eps * (sum_y + np.abs(rho * y).sum())
    assert d["u_max"] == math.sqrt(np.max(f[1] * f[1] + f[2] * f[2]))


def test_diagnostics_of_an_overflowed_lattice():
    from paper_1806_10241_gb300.solver import Solver
    params = BUILDERS["cylinder_axis"](40, 24)
    s = Solver(params, storage="fp32")
    base = random_state(params, 5)
    big = base.copy()
    big[1, 11, 20] += 1e12  # a velocity of 1e12 in row 12, where the density stays
    big[0, 12, 20] -= 1e12
    s.set_dist(big)
    d, f = s.diag(), s.fields()
    assert np.all(np.isfinite(f)) and 1e11 < np.abs(f[1]).max()
    assert d["u_max"] == math.sqrt(np.max(f[1] * f[1] + f[2] * f[2]))
    huge = base.copy()
    huge[0, 10:18, 7] = 3e38  # the column's sum leaves the FP32 range, its FP64 sum does not
    s.set_dist(huge)
    assert s.diag()["mass"] == pytest.approx(8 * 3e38, rel=1e-6)
    inf = base.copy()
    inf[0, 3, 3] = np.inf
    s.set_dist(inf)
    d = s.diag()
    assert d["mass"] == np.inf and d["status"] != 0
