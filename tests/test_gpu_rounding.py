"""Stochastic rounding of 16-bit storage: each rounding of a step is the one
that the documented random words give, word for word (the PCG hash of node and
step salt, then xorshift32 over the node's planes), on the values that an FP32
lattice computes from the same state."""
import struct

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


M32, M64 = 0xffffffff, 0xffffffffffffffff


def _words(nr, nz, pitch, step):
    """The 19 words of each column pair, [19, nz, pairs], as uint32."""
    z = (step + 0x9E3779B97F4A7C15) & M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    salt = (z ^ (z >> 31)) & M32
    u32 = np.uint32
    v = (np.arange(nz, dtype=u32)[:, None] * u32(pitch) + np.arange(0, nr + (nr & 1), 2, dtype=u32)) ^ u32(salt)
    s = v * u32(747796405) + u32(2891336453)
    w = ((s >> ((s >> u32(28)) + u32(4))) ^ s) * u32(277803737)
    w = ((w >> u32(22)) ^ w) | u32(1)
    out = []
    for _ in range(19):
        w = w ^ (w << u32(13))
        w = w ^ (w >> u32(17))
        w = w ^ (w << u32(5))
        out.append(w)
    return np.stack(out)


def _planes(blob, dtype, nr, nz, pitch):
    return np.frombuffer(blob, dtype, 19 * nz * pitch, offset=16).reshape(19, nz, pitch)[:, :, :nr]


@pytest.mark.parametrize("storage", ["fp16", "bf16"])
@pytest.mark.parametrize("name,nr,nz", [("cylinder_axis", 70, 9), ("czochralski", 129, 31), ("periodic_annulus", 65, 40)])
def test_roundings_are_those_of_the_documented_words(name, nr, nz, storage):
    from paper_1806_10241_gb300.solver import Solver
    params, step = BUILDERS[name](nr, nz), 987654321
    bits = 13 if storage == "fp16" else 16  # mantissa bits that the conversion drops
    scale = np.float32(1024 if storage == "fp16" else 1)
    low, full = Solver(params, storage=storage), Solver(params, storage="fp32")
    low.set_dist(random_state(params, 3))
    p16, p32 = -(-nr // 64) * 64, -(-nr // 32) * 32

    def values(blob):
        raw = _planes(blob, np.uint16, nr, nz, p16)
        if storage == "fp16":
            return raw.view(np.float16).astype(np.float32)
        return (raw.astype(np.uint32) << 16).view(np.float32)

    blob = low.get_state()
    start = np.zeros((19, nz, p32), np.float32)
    start[:, :, :nr] = values(blob) / scale
    fblob = bytearray(full.get_state())
    fblob[16:16 + start.nbytes] = start.tobytes()
    full.set_state(bytes(fblob))
    low.set_state(struct.pack("<q", step) + blob[8:])
    full.step(1)
    low.step(1)
    exact = _planes(full.get_state(), np.float32, nr, nz, p32) * scale
    got = values(low.get_state())
    w = _words(nr, nz, p16, step)
    r = np.stack([w, w >> np.uint32(16)], axis=-1).reshape(19, nz, -1)[:, :, :nr] & np.uint32((1 << bits) - 1)
    drop = np.uint32((1 << bits) - 1)
    want = ((np.ascontiguousarray(exact).view(np.uint32) + r) & ~drop).view(np.float32)
    normal = np.abs(exact) > 2.0 ** -14  # (FP16 drops more bits of a subnormal)
    # FP32 arithmetic may differ by a rounding between the two lattices, 2^-24 of a value whose storage unit is 2^-11
    # or 2^-8: some roundings in a thousand.  Independent words would agree on two thirds.
    assert normal.mean() > 0.9
    assert np.mean(want[normal] == got[normal]) > 0.99
