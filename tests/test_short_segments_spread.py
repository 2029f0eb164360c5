"""Short segments (n = 4, 8, 16) in launches of 1 to 8 warps per CTA: batches that
end anywhere around a warp per SM and eight, and one that gives every resident
warp more than one unit of 512 points; both directions and |X|^2 (the shared
memory is rewritten unit by unit, and |X|^2 changes its row size), every segment
against numpy's FP64 DFT."""
import numpy as np
import pytest

import siggen
from tests._util import check_guard, guard, rel_l2, tol_fp32, tol_power

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402


@pytest.mark.parametrize("n", [4, 8, 16])
@pytest.mark.parametrize("per_sm,extra", [(0, 1), (1, -1), (1, 1), (2, 1), (7, 1), (8, 0), (8, 1), (100, 3)])
def test_units_per_cta(n, per_sm, extra):
    units = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + extra
    B = units * 512 // n - 1  # a ragged last unit
    x = siggen.uniform(3200 + n, B * n).reshape(B, n)
    d = torch.from_numpy(x).cuda()
    F = np.fft.fft(x.astype(np.complex128))
    for direction, norm, out_kind in ((fs.FORWARD, fs.NORM_NONE, fs.OUT_COMPLEX),
                                      (fs.INVERSE, fs.NORM_BACKWARD, fs.OUT_COMPLEX),
                                      (fs.FORWARD, fs.NORM_NONE, fs.OUT_POWER)):
        power = out_kind == fs.OUT_POWER
        buf, y = guard(torch.empty(B, n, dtype=torch.float32 if power else torch.complex64, device="cuda"))
        plan = fs.Plan(n, B, direction, norm, out_kind=out_kind)
        plan.exec(d, out=y)
        torch.cuda.synchronize()
        plan.check()
        check_guard(buf)
        ref = np.abs(F) ** 2 if power else F if direction == fs.FORWARD else np.fft.ifft(x.astype(np.complex128))
        assert rel_l2(y.cpu().numpy(), ref) <= (tol_power(n) if power else tol_fp32(n))
