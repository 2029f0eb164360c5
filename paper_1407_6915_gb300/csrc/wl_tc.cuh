// Tensor-core lines of the lane-line four-step kernel at 256 x 256: both
// radix-16 stages of a 256-point line as 32 x 32 real products on
// mma.sync.m16n8k16 with split hi+lo 16-bit operands (tc.cuh has the method:
// Y ~ Fh Xl + Fl Xh + Fh Xh, FP32 accumulation).
//
// The DFT matrix is the A operand and eight butterflies are the columns of B,
// so that the fragments are what a lane can read and write directly, with no
// staging of operands: with g = lane / 4, t = lane % 4
//   B: lane (g, t) holds points t + 4 i, i < 4, of butterfly g (re and im are
//      neighbouring k indices), four 8-byte loads from the tile;
//   C: lane (g, t) holds bins g and g + 8 (rows g and g + 8 of a 16-row tile
//      are the re and im of one bin) of butterflies 2 t and 2 t + 1.
// A warp holds four lines of a panel, columns 2 w + {0, 1, 8, 9} (w: the warp's
// number in its panel), and runs them in eight groups of eight butterflies:
// butterfly g of group G is line 2 w + (g & 1) + 8 ((g >> 1) & 1), butterfly
// b = 2 G + (g >> 2).  So C's two butterflies are one b of two neighbouring
// lines: a 16-byte store.
//
// FP16 operands are scaled into range by a power of two taken from the
// butterfly's largest component and scaled back exactly, as dft16_tc does.  The
// four lanes of a butterfly find its exponent by two shuffles, and two more bring
// a lane those of its two output butterflies: 451 us for the 1024 segments below.
// (One maximum for the eight butterflies of a group, by a warp reduction, took
// 432 but left a quiet line beside a loud one with fewer bits, down to an error of
// 1.7e-3 at 2^-30 of its neighbour.  That maximum where the group is even and
// the shuffles else, 496; four groups' exponents in the bytes of one word, 470.)
//
// Tile rows: element (hi, lo) of a line, hi, lo < 16, is in row 16 hi + lo, its
// 16-byte chunk at (column / 2) ^ (lo & 7) ^ X(hi).  Input tiles hold point
// 16 lo + hi there (butterfly hi, point lo of its sixteen), which the tensor
// map of the input and the ring's row order provide.  Column tiles: X = 0, the
// TMA swizzle.  Row tiles: X(hi) = 4 (hi >> 3) ^ (q & 3), q = k1 / 16, the
// pattern that lets the column pass write its staged ring rows without bank
// conflicts; the ring holds the rows as they are in shared memory.  The
// exchange puts bin k of butterfly b at (k, b ^ 2 (k & 1)).  Every access is
// conflict-free but the row tiles' staged output (two-way).
//
// 1024 segments of 65536 points, FP16 hi+lo: 451 us (BF16: 376 us) against
// 1159 us on the CTA-tile kernel, whose operands, hi and lo, and results all
// pass through shared memory once more per stage.  Tensor pipe 37 % active,
// shared-memory pipe 41 %, issue 36 %: bound by latency, with two compute warps
// per scheduler.  (Sixteen warps, two to four lines: 418 and 410 us, against 439
// and 377 then.)
#pragma once
#include "tc.cuh"

namespace fftseg {

// The DFT matrix as A fragments: [row tile][k step][a0..a3], hi and lo.
struct WlTcF {
    uint32_t h[2][2][4], l[2][2][4];
    template <int S, int PREC>
    FDEV void init(int g, int t)
    {
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int kt = 0; kt < 2; ++kt)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int m = g + 8 * mt, r = t + 4 * (2 * kt + q);
                    const float c = cos16(r * m), s = (float)S * sin16(r * m);
                    float la, lb;
                    h[mt][kt][2 * q] = pack_hi<PREC>(c, -s, la, lb);  // row re(m)
                    l[mt][kt][2 * q] = pack_lo<PREC>(la, lb);
                    h[mt][kt][2 * q + 1] = pack_hi<PREC>(s, c, la, lb);  // row im(m)
                    l[mt][kt][2 * q + 1] = pack_lo<PREC>(la, lb);
                }
    }
};

// Eight butterflies: d[mt] = (re, re', im, im') of bin g + 8 mt of butterflies
// 2 t and 2 t + 1 from this lane's points x[i] = t + 4 i of butterfly g, scaled
// by sc (FP16) and the two back by inv.
template <int PREC>
FDEV void wl_tc_group(float (&d)[2][4], const float2 (&x)[4], float sc, float2 inv, const WlTcF &F)
{
    uint32_t xh[4], xl[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float la, lb;
        const float2 y = PREC == PREC_FP16 ? cscale(x[i], sc) : x[i];
        xh[i] = pack_hi<PREC>(y.x, y.y, la, lb);
        xl[i] = pack_lo<PREC>(la, lb);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) d[i >> 2][i & 3] = 0.f;
    // (products in an order that alternates between accumulators, or between
    // those of two groups, measured the same)
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
#pragma unroll
        for (int kt = 0; kt < 2; ++kt) {
            mma16816<PREC>(d[mt], F.h[mt][kt], xl[2 * kt], xl[2 * kt + 1]);
            mma16816<PREC>(d[mt], F.l[mt][kt], xh[2 * kt], xh[2 * kt + 1]);
            mma16816<PREC>(d[mt], F.h[mt][kt], xh[2 * kt], xh[2 * kt + 1]);
        }
        if constexpr (PREC == PREC_FP16) {
#pragma unroll
            for (int i = 0; i < 4; i += 2) {
                const float2 y = cmul_each(make_float2(d[mt][i], d[mt][i + 1]), inv);
                d[mt][i] = y.x;
                d[mt][i + 1] = y.y;
            }
        }
    }
}

// This warp's four lines of the panel at byte offset pb, in place in the tile
// buffer; ROWS: a row tile whose panel is q = qx mod 4.  On return d[G][mt]
// holds (re, re', im, im') of bin k + 16 (g + 8 mt), k = 2 G + (t >> 1), of
// lines 2 w + 8 (t & 1) and the next.
template <int S, int PREC, bool ROWS>
FDEV void wl_tc_line(float (&d)[8][2][4], char *Pc, uint32_t pb, int w, int g, int t, int qx, const WlTcF &F,
                     const float2 (&tw)[8][2], [[maybe_unused]] int *err)
{
    // (self-checking build: every slot of size bytes within the panel, aligned)
    auto at = [&](uint32_t off, [[maybe_unused]] uint32_t size) {
        if (!FFTSEG_CHECK(off - pb <= 32768 - size && off % size == 0, err)) off = pb;
        return Pc + off;
    };
    auto KX = [](uint32_t x) { return 128 * x + 16 * (x & 7); };  // row and chunk bits of lo
    const uint32_t X = ROWS ? (uint32_t)qx : 0u;
    const uint32_t lc = (uint32_t)(w + 4 * ((g >> 1) & 1)) ^ X, rd = pb + 2048 * (g >> 2) + 8 * (g & 1);
    const uint32_t lw = (uint32_t)(w + 4 * (t & 1)) ^ X;
    // GB groups' points and scales before their products: one wait for the tile
    // and the shuffles instead of GB (FP16: 451 us with two, 470 with four, 464
    // with eight; BF16, which has no scales: 376 with four)
    constexpr int GB = PREC == PREC_FP16 ? 2 : 4;
    auto pass = [&](uint32_t t0) {
        const uint32_t base = rd + 128 * t0 + 16 * (lc ^ t0);
#pragma unroll
        for (int G0 = 0; G0 < 8; G0 += GB) {
            float2 x[GB][4];
            [[maybe_unused]] uint32_t e[GB];  // biased exponent of the butterfly's largest component, in place
#pragma unroll
            for (int G = 0; G < GB; ++G)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    x[G][i] = *reinterpret_cast<const float2 *>(
                        at((base ^ KX(4 * i) ^ (ROWS && G0 + G >= 4 ? 64u : 0u)) + 4096u * (G0 + G), 8));
            if constexpr (PREC == PREC_FP16) {
                float m[GB];
#pragma unroll
                for (int G = 0; G < GB; ++G) {
                    m[G] = 0x1p-100f;  // (both scales are normal)
#pragma unroll
                    for (int i = 0; i < 4; ++i) m[G] = fmaxf(m[G], fmaxf(fabsf(x[G][i].x), fabsf(x[G][i].y)));
                }
#pragma unroll
                for (int G = 0; G < GB; ++G) m[G] = fmaxf(m[G], __shfl_xor_sync(0xffffffffu, m[G], 1));
#pragma unroll
                for (int G = 0; G < GB; ++G)
                    e[G] = __float_as_uint(fmaxf(m[G], __shfl_xor_sync(0xffffffffu, m[G], 2))) & 0x7f800000u;
            }
#pragma unroll
            for (int G = 0; G < GB; ++G) {
                float sc = 1.f;
                float2 inv = make_float2(1.f, 1.f);
                if constexpr (PREC == PREC_FP16) {  // 2^(13 - e), and 2^(e - 13) of the output butterflies
                    sc = __uint_as_float((267u << 23) - e[G]);
                    const uint32_t u = e[G] - (13u << 23);
                    inv = make_float2(__uint_as_float(__shfl_sync(0xffffffffu, u, 8 * t)),
                                      __uint_as_float(__shfl_sync(0xffffffffu, u, 8 * t + 4)));
                }
                wl_tc_group<PREC>(d[G0 + G], x[G], sc, inv, F);
            }
        }
    };
    pass((uint32_t)t);
    __syncwarp();  // every lane has read its points
    const uint32_t lo = (uint32_t)((t >> 1) ^ (2 * (g & 1)));
    const uint32_t wb = pb + 2048 * g + 128 * lo + 16 * (lw ^ lo);
#pragma unroll
    for (int G = 0; G < 8; ++G)
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            const float2 a = twmul<S>(make_float2(d[G][mt][0], d[G][mt][2]), tw[G][mt]);
            const float2 b = twmul<S>(make_float2(d[G][mt][1], d[G][mt][3]), tw[G][mt]);
            *reinterpret_cast<float4 *>(at((wb ^ KX(2 * G) ^ (ROWS && mt ? 64u : 0u)) + 16384u * mt, 16)) =
                make_float4(a.x, a.y, b.x, b.y);
        }
    __syncwarp();
    pass((uint32_t)(t ^ (2 * (g >> 2))));
}

}  // namespace fftseg
