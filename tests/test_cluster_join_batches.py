"""Inverse real plans of 2^14 and 2^15 samples whose join runs in the cluster kernel:
batches on either side of those where the kernel's registers per thread change (as
many segments as SMs; a half and three quarters) give a segment the same bits, and match numpy's FP64 inverse."""
import numpy as np
import pytest

import siggen
from tests._util import check_guard, guard, rel_l2, tol_fp32

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402


@pytest.mark.parametrize("log_n", [14, 15])
def test_batches(log_n):
    n = 1 << log_n
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = 2 * sms + 3
    x = siggen.uniform(3900 + log_n, B * (n // 2 + 1)).reshape(B, -1)
    d = torch.from_numpy(x).cuda()
    outs = {}
    for b in (1, 7, sms // 2, sms // 2 + 1, 3 * sms // 4, 3 * sms // 4 + 1, sms, sms + 1, B):
        plan = fs.Plan(n, b, fs.INVERSE, fs.NORM_BACKWARD, flags=fs.FLAG_REAL)
        assert plan.info()["work_bytes"] == 0
        buf, y = guard(torch.empty(b, n, dtype=torch.float32, device="cuda"))
        plan.exec(d[:b], out=y)
        torch.cuda.synchronize()
        plan.check()
        check_guard(buf)
        outs[b] = y.cpu().numpy()
    h = x.astype(np.complex128)
    h[:, 0] = h[:, 0].real
    h[:, -1] = h[:, -1].real
    assert rel_l2(outs[B], np.fft.irfft(h, n)) <= tol_fp32(n)
    for b, y in outs.items():
        np.testing.assert_array_equal(y, outs[B][:b])
