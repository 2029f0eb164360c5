"""Forward real segments of 4 to 64 samples: bin pairs one at a time up to n = 32,
in batches from there on.  Batches that end around a tile of segments, bins and
|X|^2, every segment against numpy's FP64 real DFT."""
import numpy as np
import pytest

import siggen
from tests._util import check_guard, guard, rel_l2, tol_fp32, tol_power

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402


@pytest.mark.parametrize("n", [4, 8, 16, 32, 64])
@pytest.mark.parametrize("B", [1, 2, 31, 127, 129, 256, 257, 5001])
def test_forward(n, B):
    x = np.ascontiguousarray(siggen.uniform(3400 + n, B * n).reshape(B, n).real)
    d = torch.from_numpy(x).cuda()
    F = np.fft.rfft(x.astype(np.float64))
    for power in (0, 1):
        plan = fs.Plan(n, B, fs.FORWARD, fs.NORM_ORTHO, out_kind=fs.OUT_POWER if power else fs.OUT_COMPLEX,
                       flags=fs.FLAG_REAL)
        buf, y = guard(torch.empty(B, n // 2 + 1, dtype=torch.float32 if power else torch.complex64, device="cuda"))
        plan.exec(d, out=y)
        torch.cuda.synchronize()
        plan.check()
        check_guard(buf)
        ref = np.abs(F) ** 2 / n if power else F / np.sqrt(n)
        assert rel_l2(y.cpu().numpy(), ref) <= (tol_power(n) if power else tol_fp32(n))
