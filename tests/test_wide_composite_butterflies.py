"""The composite butterflies of the Bluestein row kernel (radix 18 and 24 as coprime
products, 10 and 20 as twiddled 2 x 5 and 4 x 5), compiled for the host from the
kernels' own header against the direct DFT in double."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1407_6915_gb300", "csrc")

HARNESS = r'''
#include "engine.cuh"
#include <cmath>
#include <cstdio>
using namespace fftseg;
template <int R, class F> double err(int S, F dft_r) {
    float2 v[R]; double xr[R], xi[R];
    unsigned st = 777u + R * 7u + (S > 0);
    for (int i = 0; i < R; ++i) {
        st = st * 1103515245u + 12345u; v[i].x = (float)((st >> 8) / 16777216.0 - 0.5);
        st = st * 1103515245u + 12345u; v[i].y = (float)((st >> 8) / 16777216.0 - 0.5);
        xr[i] = v[i].x; xi[i] = v[i].y;
    }
    dft_r(v);
    double num = 0, den = 0;
    for (int k = 0; k < R; ++k) {
        double ar = 0, ai = 0;
        for (int j = 0; j < R; ++j) {
            const double ph = S * 2.0 * M_PI * (double)((j * k) % R) / R;
            ar += xr[j] * cos(ph) - xi[j] * sin(ph);
            ai += xr[j] * sin(ph) + xi[j] * cos(ph);
        }
        num += (v[k].x - ar) * (v[k].x - ar) + (v[k].y - ai) * (v[k].y - ai);
        den += ar * ar + ai * ai;
    }
    return sqrt(num / den);
}
#define T(R, f) printf("%d %.3e\n", R, fmax(err<R>(-1, [](float2 *v) { f<R, -1>(v); }), err<R>(1, [](float2 *v) { f<R, 1>(v); })));
template <int R, int S> void ab(float2 *v) { dft_ab<R / 5, 5, S>(v); }
template <int R, int S> void plain(float2 *v) { dft<R, S>(v); }
int main() {
    T(18, plain) T(24, plain) T(10, ab) T(20, ab)
    return 0;
}
'''


def test_butterflies_match_the_direct_dft(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "c.cu", tmp_path / "c"
    src.write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    errs = {int(a): float(b) for a, b in (line.split() for line in out.splitlines())}
    assert set(errs) == {10, 18, 20, 24}
    for r, e in errs.items():
        assert e < 4e-7 * r.bit_length(), (r, e)
