"""What this framework is timed on: its public calls over the lengths, batch
sizes and options that its users have.

A case is a dict of plain values.  `kind` says which call it is:
  c2c     Plan over complex segments (any length; FP32 or a tensor-core
          precision; complex or |X|^2 output)
  trip    a forward Plan, then the inverse one on its spectrum
  real    a forward real-signal Plan (FLAG_REAL)
  rtrip   a forward real-signal Plan, then the inverse one on its bins
  frames  FramePlan: overlapping windowed frames of one signal
  serve   Server: a mix of jobs of different lengths, submitted and awaited
"""
import math
import random

import numpy as np
import torch

import paper_1407_6915_gb300 as fs

NORMS = {"none": fs.NORM_NONE, "backward": fs.NORM_BACKWARD, "ortho": fs.NORM_ORTHO}
PRECISIONS = {"fp32": fs.PREC_FP32, "tc_fp16": fs.PREC_TC_FP16, "tc_bf16": fs.PREC_TC_BF16}
DIRECTIONS = {"forward": fs.FORWARD, "inverse": fs.INVERSE}
WINDOWS = {"rect": fs.WINDOW_RECT, "hann": fs.WINDOW_HANN}
SERVE_TIMEOUT_US = 30_000_000
MAX_POINTS = 1 << 27        # samples of a drawn case
MAX_CHIRP_POINTS = 1 << 25  # of a drawn case whose length has a large prime factor


def listed():
    return [
        # the smallest call: a handful of the paper's 1024-point records, as an
        # interactive program asks for them (launch latency)
        _c2c("records_few", 1024, 8),
        # one 32 MiB block of 1024-point records
        _c2c("records_block", 1024, 4096),
        # a mid-length batch with an odd count, unitary inverse
        _c2c("mid_inverse", 16384, 4001, direction="inverse", norm="ortho"),
        # the resident large batch: forward, then inverse of the spectrum
        {"name": "signal_round_trip", "kind": "trip", "n": 65536, "batch": 4096, "input": "tones"},
        # one chunk of the power-spectrum stream over 2^20-point segments
        _c2c("power_spectra", 1 << 20, 64, out="power", inp="tones"),
        # segments too long for the on-chip intermediate
        _c2c("long_segments", 1 << 22, 37),
        # the split-precision form on the tensor cores
        _c2c("tensor_core", 65536, 1024, precision="tc_fp16"),
        # real samples to their half spectrum and back (filtering in frequency)
        {"name": "real_round_trip", "kind": "rtrip", "n": 1 << 18, "batch": 501, "input": "tones"},
        # a spectrogram: half-overlapping Hann frames, |X|^2
        {"name": "spectrogram", "kind": "frames", "n": 1024, "hop": 512, "batch": 100003, "window": "hann",
         "out": "power", "input": "tones"},
        # a decimal length
        _c2c("decimal_length", 1000, 40001, direction="inverse", norm="backward"),
        # a prime length
        _c2c("prime_length", 10007, 2501),
        # a server's burst: lengths log-uniform over 2^8..2^22, both directions
        {"name": "server_burst", "kind": "serve", "mix": 5, "jobs": 24, "log_job": 24},
    ]


def _c2c(name, n, batch, direction="forward", norm="none", precision="fp32", out="complex", inp="uniform"):
    return {"name": name, "kind": "c2c", "n": n, "batch": batch, "direction": direction, "norm": norm,
            "precision": precision, "out": out, "input": inp}


def draw(rng):
    kind = rng.choice(["c2c", "c2c", "trip", "tc", "real", "rtrip", "frames", "smooth", "chirp", "serve"])
    inp = rng.choice(["uniform", "tones"])
    if kind == "serve":
        return {"kind": "serve", "mix": rng.randrange(1 << 30), "jobs": rng.randint(8, 32),
                "log_job": rng.randint(20, 24)}
    if kind in ("c2c", "trip"):
        n = 1 << rng.randint(4, 23)
    elif kind == "tc":
        n = 1 << rng.choice([12, 16, 20])
    elif kind in ("real", "rtrip"):
        n = 1 << rng.randint(8, 20)
    elif kind == "frames":
        n = 1 << rng.randint(8, 18)
    elif kind == "smooth":
        n = rng.choice([2 ** a * 3 ** b * 5 ** c * 7 ** d for a in range(10) for b in range(5) for c in range(4)
                        for d in range(3) if b + c + d and 90 <= 2 ** a * 3 ** b * 5 ** c * 7 ** d <= 4096])
    else:
        n = _log_uniform(rng, 100, 200000)
        while _smooth(n):
            n += 1
    cap = MAX_CHIRP_POINTS if kind == "chirp" else MAX_POINTS
    batch = _log_uniform(rng, 1, max(1, cap // n))
    if kind == "trip":
        return {"kind": "trip", "n": n, "batch": batch, "input": inp}
    if kind == "rtrip":
        return {"kind": "rtrip", "n": n, "batch": batch, "input": inp}
    out = rng.choice(["complex", "complex", "power"])
    if kind == "real":
        return {"kind": "real", "n": n, "batch": batch, "out": out, "input": inp}
    if kind == "frames":
        hop = rng.choice([n // 4, n // 2, n, _log_uniform(rng, n // 8, n)])
        return {"kind": "frames", "n": n, "hop": hop, "batch": batch, "window": rng.choice(["hann", "rect"]),
                "out": out, "input": inp}
    direction = rng.choice(["forward", "inverse"])
    precision = rng.choice(["tc_fp16", "tc_bf16"]) if kind == "tc" else "fp32"
    case = _c2c("", n, batch, direction, rng.choice(["none", "backward", "ortho"]), precision, out, inp)
    del case["name"]
    return case


def _log_uniform(rng, lo, hi):
    return min(hi, int(lo * math.exp(rng.random() * math.log((hi + 1) / lo))))


def _smooth(n):
    if n > 4096 and n & (n - 1):
        return False
    for p in (2, 3, 5, 7):
        while n % p == 0:
            n //= p
    return n == 1


# ------------------------------------------------------------------- inputs

def _uniform(count, dtype, gen):
    reals = count * (2 if dtype == torch.complex64 else 1)
    x = torch.rand(reals, generator=gen, device="cuda").mul_(2).sub_(1)
    return torch.view_as_complex(x.view(-1, 2)) if dtype == torch.complex64 else x


def _tones(count, dtype, seed, gen):
    """32 off-bin tones, amplitudes log-uniform on [1e-3, 1], and Gaussian noise
    of sigma 0.1; the tones as the product of a factor per 4096-sample row and
    one per column."""
    r = np.random.default_rng(seed)
    freq, phase, amp = r.random(32), r.random(32), 10.0 ** (-3 * r.random(32))
    rows, cols = -(-count // 4096), 4096
    a = torch.exp(2j * math.pi * torch.frac(torch.arange(rows, device="cuda", dtype=torch.float64)[:, None] * 4096
                                            * torch.tensor(freq, device="cuda") + torch.tensor(phase, device="cuda")))
    b = torch.exp(2j * math.pi * torch.frac(torch.tensor(freq, device="cuda")[:, None]
                                            * torch.arange(cols, device="cuda", dtype=torch.float64)))
    a = (a * torch.tensor(amp, device="cuda")).to(torch.complex64)
    b = b.to(torch.complex64)
    if dtype == torch.complex64:
        x = a @ b
        torch.view_as_real(x).add_(torch.randn((rows, cols, 2), generator=gen, device="cuda"), alpha=0.1)
    else:
        x = torch.addmm(torch.randn((rows, cols), generator=gen, device="cuda"),
                        torch.cat([a.real, -a.imag], 1), torch.cat([b.real, b.imag], 0), beta=0.1)
    return x.view(-1)[:count]


def _samples(count, dtype, kind, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    return _tones(count, dtype, seed, gen) if kind == "tones" else _uniform(count, dtype, gen)


def _input(case, seed):
    if case["kind"] == "frames":
        return _samples((case["batch"] - 1) * case["hop"] + case["n"], torch.complex64, case["input"], seed)
    dtype = torch.float32 if case["kind"] in ("real", "rtrip") else torch.complex64
    return _samples(case["batch"] * case["n"], dtype, case["input"], seed).view(case["batch"], case["n"])


def _jobs(case):
    """(n, segments, direction) of every job of a server's mix."""
    rng = random.Random(case["mix"])
    jobs = []
    for _ in range(case["jobs"]):
        e = rng.randint(8, 22)
        nseg = min(int(2 ** rng.uniform(0, 12)), max(1, 1 << max(0, case["log_job"] - e)))
        jobs.append((1 << e, nseg, rng.choice(["forward", "inverse"])))
    return jobs


def _job_inputs(case, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    return [_uniform(n * s, torch.complex64, gen).view(s, n) for n, s, _ in _jobs(case)]


# -------------------------------------------------------------------- calls

def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        x = _job_inputs(case, seed)
        state = {"kind": kind, "jobs": _jobs(case), "x": x, "out": [torch.empty_like(v) for v in x],
                 "server": fs.Server()}
        run(state)  # a server in service has its resident plans
        return state
    n, batch = case["n"], case["batch"]
    x = _input(case, seed)
    state = {"kind": kind, "x": x}
    out = fs.OUT_POWER if case.get("out") == "power" else fs.OUT_COMPLEX
    if kind == "c2c":
        state["plan"] = fs.Plan(n, batch, DIRECTIONS[case["direction"]], NORMS[case["norm"]],
                                PRECISIONS[case["precision"]], out)
    elif kind == "frames":
        state["plan"] = fs.FramePlan(n, case["hop"], batch, WINDOWS[case["window"]], out_kind=out)
    else:
        flags = 0 if kind == "trip" else fs.FLAG_REAL
        state["plan"] = fs.Plan(n, batch, fs.FORWARD, out_kind=out, flags=flags)
        if kind != "real":
            state["inverse"] = fs.Plan(n, batch, fs.INVERSE, fs.NORM_BACKWARD, flags=flags)
    cols = n // 2 + 1 if kind in ("real", "rtrip") else n
    state["out"] = torch.empty((batch, cols), device="cuda",
                               dtype=torch.float32 if out == fs.OUT_POWER else torch.complex64)
    if "inverse" in state:
        state["back"] = torch.empty_like(x)
    return state


def run(state):
    if state["kind"] == "serve":
        server = state["server"]
        torch.cuda.current_stream().synchronize()  # the server reads the inputs on streams of its own
        ids = [server.submit(x, y, n, s, DIRECTIONS[d], fs.NORM_BACKWARD if d == "inverse" else fs.NORM_NONE)
               for (n, s, d), x, y in zip(state["jobs"], state["x"], state["out"])]
        for i in ids:
            done, status = server.poll(i, SERVE_TIMEOUT_US)
            if not done or status != fs.OK:
                raise RuntimeError("job %d: done %s, status %s" % (i, done, status))
        return state["out"]
    y = state["plan"].exec(state["x"], state["out"])
    if "inverse" in state:
        return y, state["inverse"].exec(y, state["back"])
    return y


def work(case):
    kind = case["kind"]
    if kind == "serve":
        jobs = _jobs(case)
        return {"bytes": sum(16 * n * s for n, s, _ in jobs),
                "flops": sum(5 * n * s * int(math.log2(n)) for n, s, _ in jobs)}
    n, batch = case["n"], case["batch"]
    flops = 5 * n * math.log2(n) * batch
    power = case.get("out") == "power"
    if kind == "frames":
        # hop >= n reads only the frames' own samples
        read = n + (batch - 1) * min(case["hop"], n)
        return {"bytes": 8 * read + (4 if power else 8) * n * batch, "flops": flops}
    if kind in ("real", "rtrip"):
        one = (4 * n + (4 if power else 8) * (n // 2 + 1)) * batch
        return {"bytes": one * (2 if kind == "rtrip" else 1), "flops": flops / 2 * (2 if kind == "rtrip" else 1)}
    one = (8 + (4 if power else 8)) * n * batch
    return {"bytes": one * (2 if kind == "trip" else 1), "flops": flops * (2 if kind == "trip" else 1)}


# -------------------------------------------------------------------- exact

def _dft(x, direction, norm):
    """The DFT of the last axis in 64 bits, scaled as a plan of that norm does."""
    n = x.shape[-1]
    if direction == "forward":
        y = torch.fft.fft(x)
    else:
        y = torch.fft.ifft(x, norm="forward")
    if norm == "ortho":
        y *= 1 / math.sqrt(n)
    elif norm == "backward" and direction == "inverse":
        y *= 1 / n
    return y


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return [_dft(x.to(torch.complex128), d, "backward")
                for (_, _, d), x in zip(_jobs(case), _job_inputs(case, seed))]
    n, batch = case["n"], case["batch"]
    x = _input(case, seed)
    if kind == "trip":
        x = x.to(torch.complex128)
        return _dft(x, "forward", "none"), x
    if kind in ("real", "rtrip"):
        x = x.double()
        y = torch.fft.rfft(x)
        if kind == "rtrip":
            return y, x
    elif kind == "frames":
        f = x.as_strided((batch, n), (case["hop"], 1)).to(torch.complex128)
        if case["window"] == "hann":
            f *= 0.5 - 0.5 * torch.cos(2 * math.pi / n * torch.arange(n, device="cuda", dtype=torch.float64))
        y = _dft(f, "forward", "none")
    else:
        y = _dft(x.to(torch.complex128), case["direction"], case["norm"])
    if case.get("out") == "power":
        return torch.view_as_real(y).square().sum(-1)
    return y
