"""The square root of the error bounds (csrc/ef_root.cuh) against CUDA's sqrtf: bit for bit for every
argument from 1e-30 to the largest finite one; below, a unit in the last place for normal ones, at
most 1e-22 for subnormal ones and zero; infinity and NaN as they are."""
import os
import subprocess

import pytest

from paper_2511_12416_gb300 import _build

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include <cmath>
#include <limits>
#include "ef_root.cuh"
// every bit pattern from `first` on, `count` of them
__global__ void k_compare(unsigned first, unsigned count, unsigned long long* wrong) {
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < count;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const float x = __uint_as_float(first + (unsigned)i);
        if (__float_as_uint(ef::root(x)) != __float_as_uint(sqrtf(x))) atomicAdd(wrong, 1ull);
    }
}
__global__ void k_special(const float* x, float* y, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) y[i] = ef::root(x[i]);
}
int main() {
    unsigned long long* wrong;
    cudaMallocManaged(&wrong, 8);
    *wrong = 0;
    unsigned lo;
    const float tiny = 1e-30f;
    __builtin_memcpy(&lo, &tiny, 4);
    k_compare<<<1024, 256>>>(lo, 0x7f800000u - lo, wrong);
    float *x, *y;
    cudaMallocManaged(&x, 32);
    cudaMallocManaged(&y, 32);
    const float v[] = {0.f, 1e-45f, 1e-38f, 2e-38f, 9e-31f, std::numeric_limits<float>::infinity(), NAN};
    for (int i = 0; i < 7; ++i) x[i] = v[i];
    k_special<<<1, 32>>>(x, y, 7);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    printf("%llu", *wrong);
    for (int i = 0; i < 7; ++i) printf(" %.9g", y[i]);
    printf("\n");
}
"""


def test_root_against_sqrtf(tmp_path):
    (tmp_path / "m.cu").write_text(PROGRAM)
    exe = tmp_path / "m"
    subprocess.run([_build.nvcc_path(), "-O3", "-std=c++17", *_build.ARCH, "-I", _build.CSRC, str(tmp_path / "m.cu"), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120, env=os.environ)
    assert r.returncode == 0
    wrong, *special = r.stdout.split()
    assert int(wrong) == 0
    assert all(0.0 <= float(v) <= 1e-22 for v in special[:3])
    assert [float(v) for v in special[3:5]] == [pytest.approx(2e-38 ** 0.5, rel=2.0 ** -23), pytest.approx(9e-31 ** 0.5, rel=2.0 ** -23)]
    assert special[5] == "inf" and "nan" in special[6].lower()
