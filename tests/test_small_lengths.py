"""Short lengths.  The mixed-radix kernel's composite in-register butterflies (6, 9, 10, 12, 14,
15) and their compile-time rotations, compiled for the host from the kernels'
own header against the direct DFT in double, and every smooth length's schedule
on the GPU path: lengths whose stages use each of them, one and two stages, the
longest of a 2048- and a 4096-point tile, with ragged tiles."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
import siggen
from tests._util import rel_l2, tol_fp32

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1407_6915_gb300", "csrc")

HARNESS = r'''
#include "engine.cuh"
#include <cmath>
#include <cstdio>
using namespace fftseg;
template <int R, int S> double err() {
    float2 v[16]; double xr[16], xi[16];
    unsigned st = 777u + R * 7u + (S > 0);
    for (int i = 0; i < R; ++i) {
        st = st * 1103515245u + 12345u; v[i].x = (float)((st >> 8) / 16777216.0 - 0.5);
        st = st * 1103515245u + 12345u; v[i].y = (float)((st >> 8) / 16777216.0 - 0.5);
        xr[i] = v[i].x; xi[i] = v[i].y;
    }
    dft<R, S>(v);
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
#define T(R) printf("%d %.3e\n", R, fmax(err<R, -1>(), err<R, 1>()));
int main() {
    T(6) T(9) T(10) T(12) T(14) T(15)
    double w = 0;
    for (int R = 2; R <= 64; ++R)
        for (int m = 0; m < R; ++m)
            w = fmax(w, fmax(fabs(ct_cos(m, R) - cos(2 * M_PI * m / R)), fabs(ct_sin(m, R) - sin(2 * M_PI * m / R))));
    printf("0 %.3e\n", w);
    return 0;
}
'''


def test_composite_butterflies_match_the_direct_dft(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "c.cu", tmp_path / "c"
    src.write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    errs = {int(a): float(b) for a, b in (line.split() for line in out.splitlines())}
    assert set(errs) == {0, 6, 9, 10, 12, 14, 15}
    assert errs.pop(0) < 1e-14  # the compile-time cosines, in double
    for r, e in errs.items():
        assert e < 4e-7 * r.bit_length(), (r, e)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [6, 18, 24, 36, 90, 140, 210, 225, 336, 1050, 1764, 2025, 2016, 2058, 2100, 3600, 4050])
@pytest.mark.parametrize("direction", [-1, 1])
def test_every_radix_and_tile_edge(n, direction):
    torch = pytest.importorskip("torch")
    import paper_1407_6915_gb300 as fs

    spt = (2048 if n <= 2048 else 4096) // n
    for B in (1, 2 * spt + 1):
        x = siggen.uniform(4200 + n, B * n).reshape(B, n)
        y = fs.Plan(n, B, direction).exec(torch.from_numpy(x).cuda())
        torch.cuda.synchronize()
        assert rel_l2(y.cpu().numpy(), oracle.dft(x, direction)) <= tol_fp32(n), (n, B)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [16, 64, 1024, 2048])
def test_block_tile_sizes_give_the_same_bits(n):
    # batches on either side of the 2^22 points where the block kernel changes its
    # tiles: a segment's bits do not depend on them, nor on a ragged last tile
    torch = pytest.importorskip("torch")
    import paper_1407_6915_gb300 as fs

    B = (1 << 22) // n
    x = torch.view_as_complex(torch.rand((B + 1, n, 2), device="cuda").sub_(0.5))
    plan = fs.Plan(n, B + 1, fs.FORWARD, fs.NORM_ORTHO)
    large, small = plan.exec(x), plan.exec(x[:B])
    odd = plan.exec(x[:3])
    torch.cuda.synchronize()
    assert torch.equal(large[:B], small) and torch.equal(large[:3], odd)
    host = x[-2:].cpu().numpy()
    assert rel_l2(large[-2:].cpu().numpy(), oracle.fft(host, fs.FORWARD, fs.NORM_ORTHO)) <= tol_fp32(n)
