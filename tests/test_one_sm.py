"""n = 2^14 with a segment per SM (the default there) against the FP64 oracle:
fewer segments than SMs, exactly as many, one more and two rounds and one more;
all norms, |X|^2, in place; the same bits for a segment in any batch; the
requested cluster kernel still runs."""
import numpy as np
import pytest

import oracle
import siggen
from tests._util import check_guard, guard, rel_l2, tol_fp32, tol_power

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402

N = 1 << 14


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1407_6915_gb300 import build
    build.build()


def run(plan, x, dtype=torch.complex64):
    d = torch.from_numpy(x).cuda()
    buf, y = guard(torch.empty(d.shape, dtype=dtype, device="cuda"))
    plan.exec(d, out=y)
    torch.cuda.synchronize()
    plan.check()
    check_guard(buf)
    return y.cpu().numpy()


@pytest.mark.parametrize("rounds,extra", [(0, 1), (0, 7), (1, -1), (1, 0), (1, 1), (2, 1)])
@pytest.mark.parametrize("direction,norm", [(fs.FORWARD, fs.NORM_NONE), (fs.INVERSE, fs.NORM_BACKWARD),
                                            (fs.INVERSE, fs.NORM_ORTHO)])
def test_one_sm_matches_oracle(rounds, extra, direction, norm):
    B = rounds * torch.cuda.get_device_properties(0).multi_processor_count + extra
    x = siggen.tones(6200 + B, B * N).reshape(B, N)
    plan = fs.Plan(N, B, direction, norm)
    assert plan.info()["path"] == "one-sm" and plan.info()["launches_per_exec"] == 1
    got = run(plan, x)
    segs = np.unique(np.r_[0, B // 2, B - 1])
    assert rel_l2(got[segs], oracle.fft(x[segs], direction, norm)) <= tol_fp32(N)
    one = run(fs.Plan(N, 1, direction, norm), x[B - 1:])
    np.testing.assert_array_equal(one[0], got[B - 1])
    d = torch.from_numpy(x).cuda()
    plan.exec(d, out=d)  # in place
    torch.cuda.synchronize()
    np.testing.assert_array_equal(d.cpu().numpy(), got)


def test_one_sm_power_and_the_requested_cluster():
    B = 5
    x = siggen.uniform(6300, B * N).reshape(B, N)
    X = oracle.fft(x, fs.FORWARD, fs.NORM_ORTHO)
    got = run(fs.Plan(N, B, fs.FORWARD, fs.NORM_ORTHO, out_kind=fs.OUT_POWER), x, torch.float32)
    assert rel_l2(got, X.real ** 2 + X.imag ** 2) <= tol_power(N)
    plan = fs.Plan(N, B, fs.FORWARD, fs.NORM_ORTHO, flags=fs.FLAG_CLUSTER_LOG2(2))
    assert plan.info()["path"] == "cluster"
    assert rel_l2(run(plan, x), X) <= tol_fp32(N)
