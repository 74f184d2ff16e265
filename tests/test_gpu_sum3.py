"""The three-float sums of the solver's FP32 phases: many pairs a lane, of either
sign and 40 binary orders of size, against math.fsum of the same parts.  Bar: adding the same pairs in FP64 may lose 2^-53 of the sum of absolute
values at every addition; the three-float sum may lose 2^-52 of it in all."""
import math
import struct
import subprocess

import numpy as np
import pytest

from paper_2608_24348_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <cuda_runtime.h>
#include "sum3.cuh"
__global__ void k(const float *a, int per, double *out)  // [2 values][32 lanes][per][2]
{
    const unsigned lane = threadIdx.x;
    Sum3 d[2] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
    for (int v = 0; v < 2; ++v)
        for (int i = 0; i < per; ++i) {
            const float *p = a + ((v * 32 + lane) * per + i) * 2;
            sum3_add(d[v], p[0], p[1], 0.f);
        }
    const double s = warp_sum3(d, lane);
    if (lane % 16 == 0) out[lane / 16] = s;
}
int main(int argc, char **argv)
{
    const int per = atoi(argv[2]), n = 2 * 32 * per * 2;
    float *h = (float *)malloc(n * sizeof(float)), *a;
    FILE *f = fopen(argv[1], "rb");
    if (!f || fread(h, sizeof(float), n, f) != (size_t)n) return 1;
    double *o, r[2];
    if (cudaMalloc(&a, n * sizeof(float)) || cudaMalloc(&o, 2 * sizeof(double))) return 2;
    cudaMemcpy(a, h, n * sizeof(float), cudaMemcpyHostToDevice);
    k<<<1, 32>>>(a, per, o);
    if (cudaMemcpy(r, o, sizeof(r), cudaMemcpyDeviceToHost)) return 3;
    fwrite(r, sizeof(double), 2, stdout);
    return 0;
}
"""


def test_sums_of_many_pairs(tmp_path):
    src, exe, dat = tmp_path / "s.cu", tmp_path / "s", tmp_path / "d"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    rng = np.random.default_rng(3)
    for per, spread in ((1, 0), (7, 40), (500, 0), (500, 40)):
        hi = (rng.standard_normal((2, 32, per)) * 2.0 ** rng.uniform(-spread, 0, (2, 32, per))).astype(np.float32)
        lo = (hi * rng.uniform(-(2.0 ** -25), 2.0 ** -25, hi.shape)).astype(np.float32)
        np.stack([hi, lo], -1).astype(np.float32).tofile(dat)
        raw = subprocess.run([str(exe), str(dat), str(per)], check=True, capture_output=True).stdout
        got = struct.unpack("2d", raw)
        for v in range(2):
            parts = np.concatenate([hi[v].ravel(), lo[v].ravel()]).astype(np.float64)
            assert abs(got[v] - math.fsum(parts)) <= 2.0 ** -52 * np.abs(parts).sum(), (per, spread, v)
