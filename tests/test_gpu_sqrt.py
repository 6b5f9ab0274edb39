"""sqrt_and_inverse of the stress update against sqrt and 1 / sqrt.

CUDA documents rsqrt in FP64 to 1 ulp; the root is a times it, corrected once
by its remainder, so it lies within 1 ulp of sqrt(a) too. Zero, subnormals,
infinity and NaN give what sqrt and the division give. A kernel over values of
every exponent, built here from csrc/pointwise.cuh as it is.
"""
import os
import subprocess

import numpy as np
import pytest

from paper_1601_05970_gb300 import build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "cg_passes.cuh"
#include "pointwise.cuh"

__global__ void k(const double* a, double* root, double* inv, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) fftg::sqrt_and_inverse(a[i], root[i], inv[i]);
}

int main(int argc, char** argv) {
    const int n = std::atoi(argv[3]);
    std::vector<double> v(n), o(2 * (size_t)n);
    FILE* f = std::fopen(argv[1], "rb");
    if (!f || std::fread(v.data(), 8, n, f) != (size_t)n) return 2;
    std::fclose(f);
    double* d = nullptr;
    if (cudaMalloc(&d, 3 * (size_t)n * 8) != cudaSuccess) return 3;
    if (cudaMemcpy(d, v.data(), (size_t)n * 8, cudaMemcpyHostToDevice) != cudaSuccess) return 4;
    k<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * (size_t)n, n);
    if (cudaMemcpy(o.data(), d + n, 2 * (size_t)n * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 5;
    f = std::fopen(argv[2], "wb");
    if (!f || std::fwrite(o.data(), 8, 2 * (size_t)n, f) != 2 * (size_t)n) return 6;
    std::fclose(f);
    return 0;
}
"""


def test_every_exponent(tmp_path):
    (tmp_path / "t.cu").write_text(HARNESS)
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, str(tmp_path / "t.cu"), "-o",
                                                                  str(tmp_path / "t")], check=True)
    rng = np.random.default_rng(3)
    exps = np.arange(2048, dtype=np.uint64)[:, None] << np.uint64(52)
    mant = np.concatenate([rng.integers(0, 1 << 52, (2048, 60), dtype=np.uint64),
                           np.tile(np.array([0, 1, (1 << 52) - 1, 1 << 51], dtype=np.uint64), (2048, 1))], axis=1)
    a = (exps | mant).reshape(-1).view(np.float64)  # zero, subnormals, infinity and NaN among them
    a.tofile(tmp_path / "a")
    subprocess.run([str(tmp_path / "t"), str(tmp_path / "a"), str(tmp_path / "o"), str(a.size)], check=True)
    root, inv = np.fromfile(tmp_path / "o").reshape(2, -1)
    with np.errstate(all="ignore"):
        wr = np.sqrt(a)
        normal = (a >= np.finfo(np.float64).tiny) & np.isfinite(a)
        rest = 1 / wr
        wi = 1 / np.sqrt(a.astype(np.longdouble))
    assert np.array_equal(root[~normal], wr[~normal], equal_nan=True)
    assert np.array_equal(inv[~normal], rest[~normal], equal_nan=True)
    er = np.abs(root[normal] - wr[normal]) / np.spacing(wr[normal])
    ei = np.abs(inv[normal].astype(np.longdouble) - wi[normal]) / np.spacing(wi[normal].astype(np.float64))
    assert er.max() <= 1.0
    assert ei.max() <= 1.0 + 1e-9
