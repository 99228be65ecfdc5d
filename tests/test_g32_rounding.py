"""The FP32 phase's g is the FP64 Gram-Schmidt's rows rounded to floats, bit for bit,
decided on integers where no midpoint of two floats is near.

On the host: the distance that counts as near is never below the FP64 code's own error,
2^-46 of the largest field value of the site or of the entry (eight times the bound 2^-49 of
70 roundings at 2^-53, each of at most the row's scale), for every scale the integer code
takes.  On the GPU: the floats of both codes, equal in every bit, over fields whose largest
value runs from 2^-18 to 16 and whose entries span many powers of two."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1301_3460_gb300", "csrc")

HOST = r"""
#include <cstdio>
#include "lgf_fx.cuh"
using namespace lgf;
// v = 2^(62-k), largest value mx = j / 8 of the site
int main()
{
    for (int k = 0; k < 40; k += 3)
        for (int j = 1; j < 128; j++) {
            int q = 1;
            while ((1 << (q - 1)) * 8 <= j) q++;
            const fx mx = (fx)j << (61 - q - 3);
            for (int s = -1; s <= 1; s += 2) printf("%d %d %d %llu\n", k, j, q, g2f_tol(s * (1ll << (62 - k)), mx, q));
        }
}
"""

DEVICE = r"""
#include <cstdio>
#include <cstring>
#include <cstdlib>
#include <cmath>
#include <vector>
#include "lgf_kernels.cuh"
using namespace lgf;
__global__ void both(int n, const float2* f, cx<float>* a, cx<float>* b, int* safe)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float2 f0 = f[i], f1 = f[n + i], f2 = f[2 * n + i], f3 = f[3 * n + i];
    float mx = 0.f;
    for (float v : {f0.x, f0.y, f1.x, f1.y, f2.x, f2.y, f3.x, f3.y}) mx = fmaxf(mx, fabsf(v));
    cfx r[6];
    cdig rd[6];
    const int q = fx_rows_of(f0, f1, f2, f3, mx, r, rd);
    safe[i] = fx_rows_to_float(r, mx, q, a + 6 * i);
    cx<double> X[6], g[6];
    X[0] = mk<double>(1.0, f3.x);
    X[1] = mk<double>(f0.x, f0.y);
    X[2] = mk<double>(f1.x, f1.y);
    X[3] = mk<double>(-(double)f0.x, f0.y);
    X[4] = mk<double>(1.0, f3.y);
    X[5] = mk<double>(f2.x, f2.y);
    gram_schmidt01(X, g);
    for (int e = 0; e < 6; e++) b[6 * i + e] = mk<float>((float)g[e].re, (float)g[e].im);
}
int main()
{
    const int n = 1 << 20;
    std::vector<float2> f(4 * n);
    float2* df;
    cx<float>*da, *db;
    int* ds;
    cudaMalloc(&df, 4 * n * sizeof(float2));
    cudaMalloc(&da, 6 * n * sizeof(cx<float>));
    cudaMalloc(&db, 6 * n * sizeof(cx<float>));
    cudaMalloc(&ds, n * sizeof(int));
    std::vector<cx<float>> a(6 * n), b(6 * n);
    std::vector<int> s(n);
    srand(5);
    auto u = []() { return rand() / (double)RAND_MAX * 2 - 1; };
    for (int round = 0; round < 24; round++) {
        // the largest value near 2^(3 - round), the others down to 2^-span of it
        const int span = round % 4 * 6;
        for (int i = 0; i < n; i++) {
            const double top = ldexp(1.0, 3 - round % 22), big = top * (1 + 0.99 * fabs(u()));
            const double rest = fmin(top, (15.99 - big) / 7);  // the magnitudes' sum stays below 16
            float v[8];
            for (int k = 0; k < 8; k++)
                v[k] = (float)(k == i % 8 ? (u() < 0 ? -big : big) : rest * u() * exp2(-span * fabs(u())));
            for (int k = 0; k < 4; k++) f[k * n + i] = make_float2(v[2 * k], v[2 * k + 1]);
        }
        cudaMemcpy(df, f.data(), 4 * n * sizeof(float2), cudaMemcpyHostToDevice);
        both<<<n / 256, 256>>>(n, df, da, db, ds);
        cudaMemcpy(a.data(), da, 6 * n * sizeof(cx<float>), cudaMemcpyDeviceToHost);
        cudaMemcpy(b.data(), db, 6 * n * sizeof(cx<float>), cudaMemcpyDeviceToHost);
        cudaMemcpy(s.data(), ds, n * sizeof(int), cudaMemcpyDeviceToHost);
        long safe = 0, bad = 0;
        for (int i = 0; i < n; i++)
            if (s[i]) {
                safe++;
                if (memcmp(&a[6 * i], &b[6 * i], 6 * sizeof(cx<float>))) bad++;
            }
        printf("%d %ld %ld\n", round, safe, bad);
    }
    return cudaDeviceSynchronize() != cudaSuccess || cudaGetLastError() != cudaSuccess;
}
"""


def compiled(tmp_path, text):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "g32.cu", tmp_path / "g32"
    src.write_text(text)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return [[int(x) for x in line.split()] for line in r.stdout.splitlines()]


def test_tolerance_covers_the_fp64_error(tmp_path):
    rows = compiled(tmp_path, HOST)
    assert len(rows) == 14 * 127 * 2
    for k, j, q, tol in rows:
        assert 1 <= q <= 5
        # x 2^62: mx 2^-46 = j 2^13, the entry 2^(62-k-46); no more than both and the integers' error
        assert max(j << 13, (1 << 16) >> k) <= tol <= (j << 13) + (1 << 16) + (1 << (8 + q)), (k, j)


@pytest.mark.gpu
def test_floats_equal_the_fp64_rows(tmp_path):
    rows = compiled(tmp_path, DEVICE)
    assert len(rows) == 24
    for n, safe, bad in rows:
        assert bad == 0, rows
    # the integers decide for most sites whose entries are of one size
    assert all(safe > 1 << 19 for n, safe, bad in rows if n % 4 == 0 and n < 16), rows
