"""Frames of 256, 512 and 1024 points that do not overlap (hop >= n, complex bins:
the tiles) and that do (a warp at a time), on both sides of the rule and with an
odd hop, against numpy's FP64 DFT of the windowed frames."""
import numpy as np
import pytest

import siggen
from tests._util import check_guard, guard, rel_l2, tol_fp32, tol_power

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402


@pytest.mark.parametrize("n", [256, 512, 1024])
@pytest.mark.parametrize("extra", [-1, 0, 1, 44])
@pytest.mark.parametrize("B", [1, 2, 1239])
def test_frames(n, extra, B):
    hop = n + extra
    x = siggen.tones(3300 + n + extra, (B - 1) * hop + n)
    d = torch.from_numpy(x).cuda()
    w = 0.5 - 0.5 * np.cos(2 * np.pi * np.arange(n) / n)
    frames = np.lib.stride_tricks.sliding_window_view(x.astype(np.complex128), n)[::hop]
    ref = np.fft.fft(frames * w)
    for power in (0, 1):
        plan = fs.FramePlan(n, hop, B, fs.WINDOW_HANN, out_kind=fs.OUT_POWER if power else fs.OUT_COMPLEX)
        buf, y = guard(torch.empty(B, n, dtype=torch.float32 if power else torch.complex64, device="cuda"))
        plan.exec(d, out=y)
        torch.cuda.synchronize()
        plan.check()
        check_guard(buf)
        r = np.abs(ref) ** 2 if power else ref
        assert rel_l2(y.cpu().numpy(), r) <= (tol_power(n) if power else tol_fp32(n))
