"""Bluestein rows in one SM (n = 2049 .. 12288 by default, M = q 1024 points)
against the FP64 oracle: the smallest and largest n of every q, an n whose last
block is one point, odd and even n (rows off the 16-byte boundary), one row and
more rows than the grid holds, both directions, all norms and |X|^2; and the
lengths around the range that keep their other kernels."""
import math

import numpy as np
import pytest

import oracle
import siggen
from tests._util import check_guard, guard, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402

EDGES = [2049, 2559, 2561, 3070, 3073, 3583, 3586, 4093, 4097, 4607, 4609, 5120, 5121, 6144, 6145, 7168, 7169, 7680,
         7681, 8192 + 1, 9216, 9217, 10240, 10241, 12288]


def tol_blue(n):
    # three M-point FP32 transforms' worth of rounding, as for the other Bluestein forms
    return 2e-6 * (3 * math.log2(2 * n) + 3)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1407_6915_gb300 import build
    build.build()


@pytest.mark.parametrize("n", EDGES)
@pytest.mark.parametrize("direction,norm,out_kind", [(fs.FORWARD, fs.NORM_NONE, fs.OUT_COMPLEX),
                                                     (fs.INVERSE, fs.NORM_BACKWARD, fs.OUT_COMPLEX),
                                                     (fs.FORWARD, fs.NORM_ORTHO, fs.OUT_POWER)])
def test_row_kernel_matches_direct_dft(n, direction, norm, out_kind):
    for B in (1, 307):
        x = siggen.tones(5100 + n, B * n).reshape(B, n)
        plan = fs.Plan(n, B, direction, norm, out_kind=out_kind)
        info = plan.info()
        assert info["path"] == "bluestein" and info["launches_per_exec"] == 1 and info["work_bytes"] == 0
        dt = torch.float32 if out_kind == fs.OUT_POWER else torch.complex64
        buf, y = guard(torch.empty((B, n), dtype=dt, device="cuda"))
        plan.exec(torch.from_numpy(x).cuda(), out=y)
        torch.cuda.synchronize()
        plan.check()
        check_guard(buf)
        segs = np.unique(np.r_[0, B // 2, B - 1])
        bins = np.unique(np.r_[0, 1, 1023, 1024, n // 2, n - 1, np.arange(0, n, max(1, n // 61))])
        X = oracle.dft(x[segs], direction, norm, bins=bins)
        got = y.cpu().numpy()[segs][:, bins]
        if out_kind == fs.OUT_POWER:
            assert rel_l2(got, X.real ** 2 + X.imag ** 2) <= 2 * tol_blue(n), (n, B)
        else:
            assert rel_l2(got, X) <= tol_blue(n), (n, B)


def test_row_kernel_range():
    for n, m in ((2047, 4096), (12289, 32768)):
        assert fs.Plan(n, 2).info()["n1"] == m
    assert fs.Plan(10007, 2).info()["n1"] == 20480
    assert fs.Plan(10007, 2, flags=fs.FLAG_BLUESTEIN).info()["n1"] == 32768
