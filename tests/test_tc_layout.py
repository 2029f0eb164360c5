"""The tensor-core lines of the lane-line kernel (wl_tc.cuh), their shared-memory
addressing restated and run on the CPU: for column and row tiles every access
stays in the panel and is free of bank conflicts (the staged output of row
tiles two-way), a warp's exchange stays in its own lines' slots, the two
radix-16 stages give each line's DFT in the bins the kernel stores, and the
column pass's staged ring rows are what the row pass reads."""
import numpy as np
import pytest

LANES = [(g, t) for g in range(8) for t in range(4)]


def KX(x):
    return 128 * x + 16 * (x & 7)


def phases(addrs, width):
    """Largest number of accesses to one bank group over the warp's phases."""
    per = 128 // width
    worst = 0
    for p in range(0, 32, per):
        banks = {}
        for a in set(addrs[p:p + per]):
            banks.setdefault(a % 128, set()).add(a)
        worst = max(worst, max(len(v) for v in banks.values()))
    return worst


def run_line(mem, w, rows, qx, log):
    """wl_tc_line: mem maps byte offset in the panel -> complex; returns bins
    {(line, bin)} of warp w."""
    X = qx if rows else 0
    out, own = {}, set()

    def read(t_of):
        d = {}
        for G in range(8):
            pts = {}
            for i in range(4):
                addrs = []
                for g, t in LANES:
                    t0 = t_of(g, t)
                    lc = (w + 4 * ((g >> 1) & 1)) ^ X
                    base = 2048 * (g >> 2) + 8 * (g & 1) + 128 * t0 + 16 * (lc ^ t0)
                    a = (base ^ KX(4 * i) ^ (64 if rows and G >= 4 else 0)) + 4096 * G
                    assert 0 <= a < 32768 and a % 8 == 0
                    addrs.append(a)
                    own.add(a)
                    pts[(g, t + 4 * i)] = mem[a]
                assert phases(addrs, 8) == 1
            for g in range(8):  # butterfly g of group G: its 16 points in order
                d[(G, g)] = np.fft.fft([pts[(g, r)] for r in range(16)])
        return d

    d = read(lambda g, t: t)
    first = set(own)
    new = {}
    for G in range(8):
        for mt in range(2):
            addrs = []
            for g, t in LANES:
                lo = (t >> 1) ^ (2 * (g & 1))
                lw = (w + 4 * (t & 1)) ^ X
                a = ((2048 * g + 128 * lo + 16 * (lw ^ lo)) ^ KX(2 * G) ^ (64 if rows and mt else 0)) + 16384 * mt
                assert 0 <= a < 32768 and a % 16 == 0
                addrs.append(a)
                b, k = 2 * G + (t >> 1), g + 8 * mt
                for h in range(2):
                    new[a + 8 * h] = d[(G, 2 * t + h)][k] * np.exp(-2j * np.pi * b * k / 256)
            assert phases(addrs, 16) == 1
    assert set(new) == first  # in place: the warp's own slots, each once
    mem.update(new)
    d = read(lambda g, t: t ^ (2 * (g >> 2)))
    for G in range(8):
        for g, t in LANES:
            for mt in range(2):
                k, q = 2 * G + (t >> 1), g + 8 * mt
                for h in range(2):
                    out[(2 * w + 8 * (t & 1) + h, k + 16 * q)] = d[(G, 2 * t + h)][q]
    return out


@pytest.mark.parametrize("tile,p", [(0, 0), (3, 1), (7, 0)])
def test_column_then_row_tiles(tile, p):
    rng = np.random.default_rng(tile * 2 + p)
    x = rng.standard_normal((16, 256)) + 1j * rng.standard_normal((16, 256))  # lines (columns j2) of one panel
    mem = {}
    for c in range(16):
        for j in range(256):  # row 16 b + r of point 16 r + b, TMA swizzle
            row = 16 * (j % 16) + j // 16
            mem[row * 128 + 16 * ((c >> 1) ^ (row & 7)) + 8 * (c & 1)] = x[c, j]
    bins = {}
    for w in range(4):
        bins.update(run_line(mem, w, False, 0, None))
    ref = np.fft.fft(x, axis=1)
    for (c, k), v in bins.items():
        assert abs(v - ref[c, k]) < 1e-9
    assert len(bins) == 16 * 256
    # staged ring rows [q][column][16 k]
    r = 2 * tile + p
    stage = {}
    for w in range(4):
        for G in range(8):
            for mt in range(2):
                for h in range(2):
                    addrs = []
                    for g, t in LANES:
                        c0 = 2 * w + 8 * (t & 1)
                        xx = (g & 3) ^ (4 * (t & 1)) ^ (r & 7)
                        a = ((2048 * g + 128 * c0 + 16 * xx + 8 * (t >> 1)) ^ (16 * G)) + 16384 * mt + 128 * h
                        assert 0 <= a < 32768 and a not in stage
                        addrs.append(a)
                        stage[a] = (c0 + h, 2 * G + (t >> 1) + 16 * (g + 8 * mt))
                    assert phases(addrs, 8) == 1
    assert len(stage) == 4096
    # the row tile's panel q holds row 16 b + r from this column panel's row (q, b)
    for a, (c, k1) in stage.items():
        q, b = a // 2048, (a % 2048) // 128
        assert (q, b) == (k1 // 16, c)
        lc = (a % 128) // 16 ^ (r & 7) ^ 4 * (b >> 3) ^ (q & 3)
        assert (2 * lc + (a % 16) // 8) == k1 % 16


@pytest.mark.parametrize("q", range(4))
def test_row_tiles_and_their_output(q):
    rng = np.random.default_rng(q)
    x = rng.standard_normal((16, 256)) + 1j * rng.standard_normal((16, 256))
    mem = {}
    for c in range(16):
        for j in range(256):
            b, r = j % 16, j // 16
            mem[(16 * b + r) * 128 + 16 * ((c >> 1) ^ (r & 7) ^ 4 * (b >> 3) ^ q) + 8 * (c & 1)] = x[c, j]
    assert len(mem) == 4096
    bins = {}
    for w in range(4):
        bins.update(run_line(mem, w, True, q, None))
    ref = np.fft.fft(x, axis=1)
    assert len(bins) == 4096 and all(abs(v - ref[c, k]) < 1e-9 for (c, k), v in bins.items())
    seen = set()
    for w in range(4):
        for G in range(8):
            for mt in range(2):
                addrs = []
                for g, t in LANES:
                    c0, lo = 2 * w + 8 * (t & 1), t >> 1
                    a = ((2048 * g + 128 * lo + 16 * ((c0 >> 1) ^ lo)) ^ (256 * G + 16 * ((2 * G) & 7))) + 16384 * mt
                    k2 = 2 * G + (t >> 1) + 16 * (g + 8 * mt)
                    assert a == k2 * 128 + 16 * ((c0 >> 1) ^ (k2 & 7)) and a not in seen
                    seen.add(a)
                    addrs.append(a)
                assert phases(addrs, 16) <= 2
