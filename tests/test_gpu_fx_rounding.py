"""Integer roundings of the fixed-point kernels against the hardware's conversions, equal in every
value: doubles onto the grid 2^-61, grid values to the nearest double, subnormal cotangents.
Random mantissas at every exponent of the range, ties and their neighbours, zeros, one."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1301_3460_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "lgf_fx.cuh"
using namespace lgf;
__device__ unsigned long long mix(unsigned long long x)
{
    x += 0x9e3779b97f4a7c15ull;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
    return x ^ (x >> 31);
}
__global__ void check(unsigned long long* bad)
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    // a double of magnitude 2^(-70 .. 0]: random mantissa, or few bits, so that ties occur
    const unsigned long long r = mix(i), r2 = mix(r);
    const int ex = 1023 - (int)(r2 % 71);
    unsigned long long man = r & 0xfffffffffffffull;
    if (i & 1) man &= ~((1ull << (r2 >> 8) % 53) - 1);       // trailing zeros: ties
    if ((i & 6) == 6) man |= (1ull << (r2 >> 16) % 53) - 1;  // trailing ones: just below one
    if (ex == 1023) man = 0;
    double x = __longlong_as_double((long long)((r >> 63) << 63 | (unsigned long long)ex << 52 | man));
    if (i == 0) x = 0.0;
    if (i == 1) x = -0.0;
    if (i == 2) x = __longlong_as_double(1);
    if (d2fx_rn<61>(x) != __double2ll_rn(x * 0x1p61)) atomicAdd(bad, 1ull);
    // a value x 2^62 of any size up to one
    fx v = (fx)(r2 >> 2 >> (r % 62));
    if (v > 1ll << 62) v = 1ll << 62;
    if (i & 8) v &= ~((1ll << (r >> 8) % 12) - 1);
    if (i & 16) v |= 1ll << (r >> 12) % 12;
    if (i & 32) v = -v;
    if (fx_round_double(v) != __double2ll_rn(__ll2double_rn(v) * 0.5)) atomicAdd(bad + 1, 1ull);
    // x 2^(60-e) toward zero, subnormals among the values (e = -1022: as large as they get)
    const int e = -1022 + (int)(r2 % 40);
    const double s = __longlong_as_double((long long)((r >> 63) << 63 | (r >> (12 + (r2 >> 32) % 50))));
    const double up = scalbn(s, 1000);  // exact: s is subnormal
    if (d2fx_rel(s, e) != __double2ll_rz(scalbn(up, 60 - e - 1000))) atomicAdd(bad + 2, 1ull);
}
int main()
{
    unsigned long long *d, h[3];
    cudaMalloc(&d, sizeof h);
    cudaMemset(d, 0, sizeof h);
    check<<<1 << 16, 256>>>(d);
    if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%llu %llu %llu\n", h[0], h[1], h[2]);
    return 0;
}
"""


def test_roundings_equal_the_hardware_conversions(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "rounding.cu", tmp_path / "rounding"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.split() == ["0", "0", "0"]
