"""Tensor-core lines at n = 2^16 (wl_tc.cuh).

Lines of very different magnitude side by side in FP16: the even columns of the
256 x 256 segment hold one loud pair of points (rows 0 and 128, equal, so that
their column DFT is exactly zero at odd k1), the odd columns quiet noise over
all rows.  The odd rows k1 of the row pass are then quiet lines beside loud
ones, and a scale shared between lines shows in their error.

Bound: the split keeps 22 bits of a butterfly's largest component, 2^-22 per
stage; four stages add as roots of squares, and a largest component is at most
4 times a butterfly's root mean square: 4 * 2 * 2^-22."""
import numpy as np
import pytest

import oracle
import siggen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402

N, B = 1 << 16, 3


@pytest.mark.parametrize("log_quiet", [-4, -8, -9, -20, -30])
def test_quiet_lines_beside_loud_ones(log_quiet):
    x = np.zeros((B, 256, 256), np.complex64)
    x[:, :, 1::2] = siggen.uniform(3500, B * 256 * 128).reshape(B, 256, 128) * np.float32(2.0 ** log_quiet)
    loud = siggen.uniform(3501, B * 128).reshape(B, 128)
    x[:, 0, 0::2] = x[:, 128, 0::2] = loud
    x = x.reshape(B, N)
    ref = oracle.fft(x).reshape(B, 256, 256)[:, :, 1::2]  # [segment][k2][odd k1]

    def errors(flags):
        plan = fs.Plan(N, B, fs.FORWARD, precision=fs.PREC_TC_FP16, flags=flags)
        y = plan.exec(torch.from_numpy(x).cuda())
        torch.cuda.synchronize()
        plan.check()
        d = y.cpu().numpy().reshape(B, 256, 256)[:, :, 1::2] - ref
        return np.linalg.norm(d, axis=1) / np.linalg.norm(ref, axis=1)  # per line

    lanes, tiles = errors(0), errors(fs.FLAG_FOURSTEP_TILES)
    assert lanes.max() <= 8 * 2.0 ** -22, (lanes.max(), tiles.max())
    assert lanes.max() <= 1.25 * tiles.max(), (lanes.max(), tiles.max())
