"""Mixed-radix lengths of one stage (a whole segment in a thread, n = 3 .. 15): the
bins leave through the tile.  Batches that end anywhere in a tile or start one on
an odd point, both directions, |X|^2, in place, every segment against numpy's
FP64 DFT."""
import numpy as np
import pytest

import siggen
from tests._util import check_guard, guard, rel_l2, tol_fp32, tol_power

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402


@pytest.mark.parametrize("n", [3, 5, 6, 7, 9, 10, 12, 14, 15])
@pytest.mark.parametrize("tiles", [0, 1, 3, 1300])
def test_one_stage(n, tiles):
    spt = 2048 // n
    for B in ({1, 2, spt - 1} if tiles == 0 else {tiles * spt, tiles * spt + 1}):
        x = siggen.uniform(3800 + n, B * n).reshape(B, n)
        d = torch.from_numpy(x).cuda()
        wide = x.astype(np.complex128)
        F = np.fft.fft(wide)
        for direction, norm, out_kind in ((fs.FORWARD, fs.NORM_ORTHO, fs.OUT_COMPLEX),
                                          (fs.INVERSE, fs.NORM_BACKWARD, fs.OUT_COMPLEX),
                                          (fs.FORWARD, fs.NORM_NONE, fs.OUT_POWER)):
            power = out_kind == fs.OUT_POWER
            buf, y = guard(torch.empty(B, n, dtype=torch.float32 if power else torch.complex64, device="cuda"))
            plan = fs.Plan(n, B, direction, norm, out_kind=out_kind)
            plan.exec(d, out=y)
            torch.cuda.synchronize()
            plan.check()
            check_guard(buf)
            ref = np.abs(F) ** 2 if power else F / np.sqrt(n) if direction == fs.FORWARD else np.fft.ifft(wide)
            assert rel_l2(y.cpu().numpy(), ref) <= (tol_power(n) if power else tol_fp32(n)), (n, B)
            if not power:
                z = d.clone()
                plan.exec(z, out=z)
                assert torch.equal(z, y)
