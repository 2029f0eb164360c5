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
from tests._util import TOL_TC, check_guard, guard, rel_l2
from tests.test_debug_build import dbg, run_debug  # noqa: F401

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402

N, B = 1 << 16, 3
PRECS = [fs.PREC_TC_FP16, fs.PREC_TC_BF16]


def test_power_staging_is_the_output_box():
    # every float of rows k2 x 32 lines once, in the box's 128-byte swizzle
    seen = {}
    for tid in range(256):
        lane, tp, w = tid % 32, tid >> 7, (tid >> 5) & 3
        g, t = lane >> 2, lane & 3
        c = 16 * tp + 2 * w + 8 * (t & 1)
        for G in range(8):
            for mt in range(2):
                k2 = 2 * G + (t >> 1) + 16 * (g + 8 * mt)
                off = k2 * 128 + (((c >> 2) ^ (k2 & 7)) << 4) + (c & 3) * 4
                assert off % 8 == 0
                for h in range(2):
                    assert off + 4 * h not in seen
                    seen[off + 4 * h] = (k2, c + h)
    assert len(seen) == 8192 and max(seen) < 32768
    for off, (k2, c) in seen.items():
        assert (off // 128, (((off % 128) // 16) ^ (k2 & 7)) * 4 + off % 16 // 4) == (k2, c)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("chunk_mb", [None, 1])
def test_outputs_norms_and_ragged_batches(prec, chunk_mb, monkeypatch):
    # a ring of 6 segments with 1 MiB chunks: 23 segments cycle it
    if chunk_mb:
        monkeypatch.setenv("FFTSEG_WL_CHUNK_MB", str(chunk_mb))
    nb = 23
    x = siggen.tones(3510, nb * N).reshape(nb, N)
    d = torch.from_numpy(x).cuda()
    for direction, norm in ((fs.FORWARD, fs.NORM_ORTHO), (fs.INVERSE, fs.NORM_BACKWARD)):
        ref = oracle.fft(x, direction, norm)
        for nseg in (nb, 7):
            plan = fs.Plan(N, nb, direction, norm, precision=prec)
            buf, y = guard(torch.empty(nseg, N, dtype=torch.complex64, device="cuda"))
            plan.exec(d[:nseg], out=y)
            z = d[:nseg].clone()
            plan.exec(z, out=z)
            torch.cuda.synchronize()
            plan.check()
            check_guard(buf)
            assert rel_l2(y.cpu().numpy(), ref[:nseg]) <= TOL_TC
            assert torch.equal(z, y)
            plan = fs.Plan(N, nb, direction, norm, precision=prec, out_kind=fs.OUT_POWER)
            buf, p = guard(torch.empty(nseg, N, dtype=torch.float32, device="cuda"))
            plan.exec(d[:nseg], out=p)
            torch.cuda.synchronize()
            plan.check()
            check_guard(buf)
            assert rel_l2(p.cpu().numpy(), np.abs(ref[:nseg]) ** 2) <= 2 * TOL_TC


@pytest.mark.gpu
@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("direction", [fs.FORWARD, fs.INVERSE])
def test_checked_build(dbg, prec, direction):  # noqa: F811
    nb = 70
    x = torch.from_numpy(siggen.tones(3520, nb * N).reshape(nb, N)).cuda()
    got = run_debug(dbg, lambda h: dbg.fftseg_plan_create(h, N, nb, direction, fs.NORM_NONE, prec, 0, 0), x, (nb, N))
    ref = fs.Plan(N, nb, direction, precision=prec).exec(x)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(got, ref.cpu().numpy())


@pytest.mark.gpu
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
