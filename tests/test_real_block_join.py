"""Inverse real-signal plans of n <= 8192 samples: the join fused into the block
kernel's tiles (one launch, no intermediate), against the FP64 oracle.

Bins of a segment: n/2 + 1, an odd number (n >= 4), so that tiles of one
segment start at odd bins and the batch ends on an odd bin for odd segment
counts; the imaginary parts of X[0] and X[n/2] must not enter.
"""
import numpy as np
import pytest

import oracle
import siggen
from tests._util import check_guard, guard, rel_l2, tol_fp32

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402


@pytest.mark.parametrize("log_n", range(2, 14))
@pytest.mark.parametrize("nseg", [1, 2, 3, 609, 1218])
def test_join_in_tiles(log_n, nseg):
    n = 1 << log_n
    B = nseg
    X = siggen.tones(40 + log_n, B * (n // 2 + 1)).reshape(B, n // 2 + 1)
    plan = fs.Plan(n, B, fs.INVERSE, fs.NORM_BACKWARD, flags=fs.FLAG_REAL)
    info = plan.info()
    assert info["launches_per_exec"] == 1 and info["work_bytes"] == 0, info
    buf, got = guard(torch.empty(B, n, dtype=torch.float32, device="cuda"))
    d = torch.from_numpy(X).cuda()
    plan.exec(d, out=got)
    torch.cuda.synchronize()
    plan.check()
    check_guard(buf)
    ref = oracle.irfft(X, n, fs.NORM_BACKWARD)
    assert rel_l2(got.cpu().numpy(), ref) <= tol_fp32(n)
    # a batch's bits do not depend on the segments beside them
    one = fs.Plan(n, 1, fs.INVERSE, fs.NORM_BACKWARD, flags=fs.FLAG_REAL)
    last = one.exec(d[B - 1:].clone())
    assert torch.equal(last.view(-1), got[B - 1])
