"""Segments of 2 to 16 points, a warp's 512 points at a time from n = 4 on: batches
that end anywhere in a warp's points, both directions, in place, |X|^2, against
numpy's FP64 DFT.

Bound: 16-point butterflies have four levels; the library's FP32 bound
2e-6 log2(n) covers them, per batch."""
import numpy as np
import pytest

import siggen
from tests._util import check_guard, guard, rel_l2, tol_fp32, tol_power

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402


@pytest.mark.parametrize("n", [2, 4, 8, 16])
@pytest.mark.parametrize("points", [1, 3, 31, 33, 511, 513, 40000])
def test_short(n, points):
    B = max(1, points // n) | 1
    x = siggen.uniform(3100 + n, B * n).reshape(B, n)
    d = torch.from_numpy(x).cuda()
    F, I = np.fft.fft(x.astype(np.complex128)), np.fft.ifft(x.astype(np.complex128))
    for direction, norm, ref in ((fs.FORWARD, fs.NORM_NONE, F), (fs.INVERSE, fs.NORM_BACKWARD, I)):
        plan = fs.Plan(n, B, direction, norm)
        buf, y = guard(torch.empty(B, n, dtype=torch.complex64, device="cuda"))
        plan.exec(d, out=y)
        torch.cuda.synchronize()
        plan.check()
        check_guard(buf)
        assert rel_l2(y.cpu().numpy(), ref) <= tol_fp32(n)
        z = d.clone()
        plan.exec(z, out=z)
        assert torch.equal(z, y)
    plan = fs.Plan(n, B, fs.FORWARD, out_kind=fs.OUT_POWER)
    buf, p = guard(torch.empty(B, n, dtype=torch.float32, device="cuda"))
    plan.exec(d, out=p)
    torch.cuda.synchronize()
    check_guard(buf)
    assert rel_l2(p.cpu().numpy(), np.abs(F) ** 2) <= tol_power(n)
