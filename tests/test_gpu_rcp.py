"""The FP64 step's reciprocal against the correctly rounded 1 / r: over the
densities of a lattice and over the radii that it takes too."""
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include <cuda_runtime.h>
#include "lb_rcp.cuh"
__global__ void k(const double *r, double *x, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = rcp1(r[i]);
}
int main(int, char **argv)
{
    std::vector<double> r(1 << 18);
    FILE *f = std::fopen(argv[1], "rb");
    const int n = (int)std::fread(r.data(), 8, r.size(), f);
    std::fclose(f);
    double *d, *x;
    if (cudaMalloc(&d, 8 * r.size()) != cudaSuccess || cudaMalloc(&x, 8 * r.size()) != cudaSuccess) return 1;
    cudaMemcpy(d, r.data(), 8 * (size_t)n, cudaMemcpyHostToDevice);
    k<<<(n + 255) / 256, 256>>>(d, x, n);
    if (cudaMemcpy(r.data(), x, 8 * (size_t)n, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    f = std::fopen(argv[2], "wb");
    std::fwrite(r.data(), 8, n, f);
    std::fclose(f);
    return 0;
}
"""


def test_reciprocal_is_the_correctly_rounded_one(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_10241_gb300 import build
    src, exe = tmp_path / "rcp.cu", tmp_path / "rcp"
    src.write_text(PROGRAM)
    subprocess.run([build.NVCC, *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    rng = np.random.default_rng(0)
    n = 1 << 16
    r = np.concatenate([rng.uniform(0.5, 1.75, n), np.exp(rng.uniform(np.log(0.5), np.log(2.0 ** 20), n)),
                        np.arange(n) + 0.5, np.array([0.5, 1.0, 1.5, 2.0 ** 20 + 0.5, 1e-30, 1e30])])
    r.tofile(tmp_path / "in")
    subprocess.run([str(exe), str(tmp_path / "in"), str(tmp_path / "out")], check=True)
    x = np.fromfile(tmp_path / "out")
    # the iteration leaves 1e-26 of the value where half a rounding is 1e-16: another result than the correctly rounded
    # one takes a tie to within 1e-10 of a rounding
    assert np.mean(x != 1.0 / r) < 1e-5
    assert np.max(np.abs(x * r - 1.0)) < 2.0 ** -52
