"""The integer codelets of the fixed-point transforms on the host, against a direct DFT in
extended precision: every length the kernels use, random values, constants and
alternating signs at the largest magnitude a pass admits.

Bound: every product rounds once (half a unit) after a root known to half a unit of
2^-62 and a dropped term below 1.3 units; at most log2(L) products lie on a path, each
error growing like the square root of the points still to be summed.  8 units covers
the longest codelet (measured: 5)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1301_3460_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "lgf_dft.cuh"
using namespace lgf;
template <int N, bool INV> double worst()
{
    const long double pi = 3.14159265358979323846264338327950288L;
    int c = 0;
    while ((1 << c) < N) c++;
    double e = 0;
    for (int rep = 0; rep < 60; rep++) {
        cx<fx> v[N];
        long double re[N], im[N];
        for (int i = 0; i < N; i++) {
            double a = rand() / (double)RAND_MAX * 2 - 1, b = rand() / (double)RAND_MAX * 2 - 1;
            if (rep == 0) a = b = 1.0;
            if (rep == 1) a = b = (i & 1) ? -1.0 : 1.0;
            v[i] = cx<fx>{(fx)ldexp(a, 62 - c), (fx)ldexp(b, 62 - c)};
            re[i] = (long double)v[i].re;
            im[i] = (long double)v[i].im;
        }
        dft<fx, N, INV>(v);
        for (int k = 0; k < N; k++) {
            long double sr = 0, si = 0;
            for (int j = 0; j < N; j++) {
                const long double t = 2 * pi * ((j * k) % N) / N, wr = cosl(t), wi = INV ? sinl(t) : -sinl(t);
                sr += re[j] * wr - im[j] * wi;
                si += re[j] * wi + im[j] * wr;
            }
            e = fmax(e, fmax(fabs((double)((long double)v[k].re - sr)), fabs((double)((long double)v[k].im - si))));
        }
    }
    return e;
}
template <int N> void row() { printf("%d %g %g\n", N, worst<N, false>(), worst<N, true>()); }
int main() { row<3>(); row<4>(); row<6>(); row<8>(); row<12>(); row<16>(); row<24>(); row<32>(); }
"""


def test_codelets_against_direct_dft(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "codelets.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "codelets"
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [line.split() for line in out.splitlines()]
    assert len(rows) == 8
    for n, fwd, inv in rows:
        assert float(fwd) < 8 and float(inv) < 8, (n, fwd, inv)
