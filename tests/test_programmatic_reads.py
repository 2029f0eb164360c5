"""Kernels launched with programmatic stream serialization start while the
previous kernel of the stream still runs, so the data they read may be written
while they are resident: the read-only path (__ldg), defined only for memory
that nothing writes during a kernel, may serve their plan tables and nothing
else.  Checked on the sources, and on the GPU for frames of a signal that an
in-place plan rewrites between two frame plans on one stream."""
import glob
import os
import re

import pytest

import siggen

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1407_6915_gb300", "csrc")
TABLES = {"a.tw", "a.tw1", "a.tw2", "a.bhat", "a.w", "a.twL", "a.twW", "a.window", "tw"}  # plan tables, complete before a plan is returned


def kernels():
    """(name, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            src = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__", src):
            start = src.index("{", m.start())
            depth, end = 0, start
            while True:
                depth += (src[end] == "{") - (src[end] == "}")
                end += 1
                if depth == 0:
                    break
            head = src[m.start():start]
            yield re.findall(r"(k_\w+)\s*\(", head)[-1], src[start:end]


def test_programmatic_kernels_read_only_tables_through_ldg():
    found = {name: body for name, body in kernels() if "grid_dependency_wait" in body}
    assert {"k_block", "k_short", "k_mixed", "k_block_r2c", "k_block_c2r", "k_warp_frames", "k_one_sm",
            "k_blue_row"} <= set(found)
    for name, body in found.items():
        for arg in re.findall(r"__ldg\(\s*&?([\w.]+)", body):
            assert arg in TABLES, (name, arg)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [256, 512, 1024])
@pytest.mark.parametrize("between", [16, 1024])
def test_frames_of_a_signal_rewritten_in_place(n, between):
    torch = pytest.importorskip("torch")
    import paper_1407_6915_gb300 as fs

    N = 1 << 17
    hop = n // 2
    F = (N - n) // hop + 1
    x0 = torch.from_numpy(siggen.uniform(3600 + n, N)).cuda()
    frames = fs.FramePlan(n, hop, F, fs.WINDOW_HANN, out_kind=fs.OUT_POWER)
    plan = fs.Plan(between, N // between, fs.FORWARD, fs.NORM_ORTHO)

    def chain(sync):
        x = x0.clone()
        outs = [torch.empty(F, n, dtype=torch.float32, device="cuda") for _ in range(6)]
        torch.cuda.synchronize()
        for y in outs:
            frames.exec(x, out=y)
            if sync:
                torch.cuda.synchronize()
            plan.exec(x.view(-1, between), out=x.view(-1, between))
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return outs

    ref = chain(True)
    for _ in range(20):
        for got, want in zip(chain(False), ref):
            assert torch.equal(got, want)


@pytest.mark.gpu
@pytest.mark.parametrize("n,B", [(1 << 14, 1), (1 << 14, 40), (1 << 14, 90), (10007, 1), (10007, 40), (2049, 90),
                                 (12281, 9)])
def test_chains_of_small_batches(n, B):
    # every call reads what the call before wrote, a few segments and more than
    # are launched programmatically: the same bits as with a wait between calls
    torch = pytest.importorskip("torch")
    import paper_1407_6915_gb300 as fs

    a0 = torch.from_numpy(siggen.uniform(3700 + n, B * n).reshape(B, n)).cuda()
    plans = [fs.Plan(n, B, d, fs.NORM_ORTHO) for d in (fs.FORWARD, fs.INVERSE)]
    power = fs.Plan(n, B, fs.FORWARD, fs.NORM_ORTHO, out_kind=fs.OUT_POWER)

    def chain(sync):
        a, b = a0.clone(), torch.empty_like(a0)
        p = [torch.empty((B, n), dtype=torch.float32, device="cuda") for _ in range(4)]
        torch.cuda.synchronize()
        for i in range(4):
            for plan, src, dst in ((plans[0], a, b), (power, b, p[i]), (plans[1], b, a), (plans[0], a, b),
                                   (plans[0], b, a)):
                plan.exec(src, out=dst)
                if sync:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        for plan in plans + [power]:
            plan.check()
        return [a, b] + p

    ref = chain(True)
    for _ in range(10):
        for got, want in zip(chain(False), ref):
            assert torch.equal(got, want)
