"""Mixed-radix tiles that start or end on an odd point: odd lengths in odd
batches (tiles copied in from the neighbouring even points, the last point of
the batch by itself), in either tile size, against the FP64 oracle's direct DFT
within the FP32 bound, in place and out of place."""
import numpy as np
import pytest

import oracle
import siggen
from tests._util import check_guard, guard, rel_l2, tol_fp32

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402


@pytest.mark.parametrize("n", [3, 5, 45, 105, 625, 875, 1029, 1225, 2025, 2187, 3125, 3675, 1536, 3072])
@pytest.mark.parametrize("B", [1, 2, 3, 611])
def test_odd_tiles(n, B):
    x = siggen.tones(2900 + n, B * n).reshape(B, n)
    plan = fs.Plan(n, B, fs.FORWARD)
    d = torch.from_numpy(x).cuda()
    buf, y = guard(torch.empty(B, n, dtype=torch.complex64, device="cuda"))
    plan.exec(d, out=y)
    torch.cuda.synchronize()
    plan.check()
    check_guard(buf)
    s = np.unique([0, B // 2, B - 1])
    got, ref = y.cpu().numpy()[s], oracle.dft(x[s], fs.FORWARD, fs.NORM_NONE)
    for g, r in zip(got, ref):
        assert rel_l2(g, r) <= tol_fp32(n)
    plan.exec(d, out=d)
    assert torch.equal(d, y)
