"""Batches in which every resident warp or CTA takes several units one after the
other, so that its shared memory is rewritten: overlapping frames of 256, 512 and
1024 points (a warp at a time), every frame against numpy's FP64 DFT of the
windowed frame; and n = 32 on both sides of the batch where the block kernel
changes its tiles, the same bits for a segment."""
import numpy as np
import pytest

import siggen
from tests._util import check_guard, guard, rel_l2, tol_fp32, tol_power

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402


@pytest.mark.parametrize("n", [256, 512, 1024])
@pytest.mark.parametrize("power", [0, 1])
def test_warp_frames(n, power):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    F = 3 * 16 * sms * (1024 // n) + 5  # three units for each of 16 warps per SM
    hop = n // 2 + 1
    x = siggen.tones(3950 + n, (F - 1) * hop + n)
    w = 0.5 - 0.5 * np.cos(2 * np.pi * np.arange(n) / n)
    plan = fs.FramePlan(n, hop, F, fs.WINDOW_HANN, out_kind=fs.OUT_POWER if power else fs.OUT_COMPLEX)
    buf, y = guard(torch.empty(F, n, dtype=torch.float32 if power else torch.complex64, device="cuda"))
    plan.exec(torch.from_numpy(x).cuda(), out=y)
    torch.cuda.synchronize()
    plan.check()
    check_guard(buf)
    frames = np.lib.stride_tricks.sliding_window_view(x, n)[::hop]
    got = y.cpu().numpy()
    for f0 in range(0, F, 4096):
        ref = np.fft.fft(frames[f0:f0 + 4096].astype(np.complex128) * w)
        ref = np.abs(ref) ** 2 if power else ref
        assert rel_l2(got[f0:f0 + 4096], ref) <= (tol_power(n) if power else tol_fp32(n))


@pytest.mark.parametrize("direction", [fs.FORWARD, fs.INVERSE])
def test_block_tiles_of_n_32(direction):
    n = 32
    B = (1 << 22) // n
    x = torch.view_as_complex(torch.rand((B + 1, n, 2), device="cuda").sub_(0.5))
    plan = fs.Plan(n, B + 1, direction, fs.NORM_ORTHO)
    large, small, odd = plan.exec(x), plan.exec(x[:B]), plan.exec(x[:3])
    torch.cuda.synchronize()
    assert torch.equal(large[:B], small) and torch.equal(large[:3], odd)
    host = x[-2:].cpu().numpy().astype(np.complex128)
    ref = np.fft.fft(host, norm="ortho") if direction == fs.FORWARD else np.fft.ifft(host, norm="ortho")
    assert rel_l2(large[-2:].cpu().numpy(), ref) <= tol_fp32(n)
