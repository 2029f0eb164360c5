"""The mixed-radix schedules of every length the path takes, found by the kernel's own
host code (no GPU): the radices multiply to n, no schedule has fewer stages, the
tile holds a segment, other lengths are refused; and the search asks its cost
model about a stage of given radices before it once, not once per schedule."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1407_6915_gb300", "csrc")
RADICES = (2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 15, 16)

HARNESS = r'''
static long g_model;
#define FFTSEG_COUNT_STAGE_MODEL ++g_model
#include "k_mixed.cu"
#include <cstdio>
namespace fftseg { int device_sm_count() { return 152; } }
int main() {
    for (int n = 2; n <= 4200; ++n) {
        int s, r[16], tile;
        g_model = 0;
        if (!fftseg::mixed_schedule(n, &s, r, &tile)) continue;
        printf("%d %d %ld", n, tile, g_model);
        for (int i = 0; i < s; ++i) printf(" %d", r[i]);
        printf("\n");
    }
    return 0;
}
'''


def smooth(n):
    for p in (2, 3, 5, 7):
        while n % p == 0:
            n //= p
    return n == 1


def test_every_schedule(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "s.cu", tmp_path / "s"
    src.write_text(HARNESS)
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    fewest = {1: 0}
    for n in range(2, 4097):  # by dynamic programming over divisors
        best = min((fewest[n // r] + 1 for r in RADICES if n % r == 0 and n // r in fewest), default=None)
        if best:
            fewest[n] = best
    seen = set()
    for line in out.splitlines():
        n, tile, model, *radix = map(int, line.split())
        seen.add(n)
        prod = 1
        for r in radix:
            assert r in RADICES
            prod *= r
        assert prod == n and len(radix) == fewest[n] and n <= tile and tile in (2048, 4096)
        # stages: a radix after a divisor of n, the last or not, in one of two tiles
        divisors = sum(n % d == 0 for d in range(1, n + 1))
        assert model <= 4 * divisors * len(RADICES) and model <= 400, (n, model)
    assert seen == {n for n in range(2, 4097) if smooth(n)}
