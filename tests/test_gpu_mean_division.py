"""The division behind the tile means of the kernels that keep x on chip (one Newton step with an exact remainder instead of
the general division): the function itself, compiled into a small program, against IEEE division for every significand and every
count of elements that a tile can have, and over all exponents, signs and special values."""
import subprocess

import pytest

from paper_2208_04187_b200 import build

PROGRAM = r"""
#include "halves.cuh"
#include <cstdio>
#include <cstring>
// sums whose upper bits are `high` and whose 23 significand bits run over all values in steps of `step`, by the counts [3, 256]
__global__ void compare(unsigned high, unsigned step, unsigned long long* wrong) {
    unsigned long long bad = 0;
    for (unsigned s = (blockIdx.x * blockDim.x + threadIdx.x) * step; s < (1u << 23); s += gridDim.x * blockDim.x * step) {
        const float sum = __uint_as_float(high << 23 | s);
        for (unsigned c = 3; c <= 256; ++c) {
            const float cnt = (float)c, rcp = __fdiv_rn(1.0f, cnt);
            const float a = divk::div_by_count(sum, cnt, rcp), b = __fdiv_rn(sum, cnt);
            if (__float_as_uint(a) != __float_as_uint(b) && !(a != a && b != b)) ++bad;
        }
    }
    if (bad) atomicAdd(wrong, bad);
}
int main() {
    unsigned long long* wrong;
    if (cudaMallocManaged(&wrong, sizeof(*wrong)) != cudaSuccess) return 2;
    *wrong = 0;
    compare<<<592, 256>>>(127u, 1u, wrong);                                     // every significand in [1, 2)
    if (cudaDeviceSynchronize() != cudaSuccess) return 3;
    const unsigned long long ones = *wrong;
    for (unsigned high = 0; high < 512u; ++high) compare<<<148, 256>>>(high, 509u, wrong);      // both signs, every exponent, subnormals, infinities, NaN
    if (cudaDeviceSynchronize() != cudaSuccess) return 4;
    printf("%llu %llu", ones, *wrong - ones);
    return 0;
}
"""


@pytest.mark.gpu
def test_mean_division_is_ieee_division(tmp_path):
    src = tmp_path / "t.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    flags = [f for f in build.NVCC_FLAGS if f not in ("-Xptxas", "-v", "-lineinfo")]
    subprocess.run([build._nvcc()] + flags + ["-I" + build.CSRC, str(src), "-o", exe], check=True, capture_output=True, text=True, timeout=600)
    got = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    assert got.split() == ["0", "0"], got
