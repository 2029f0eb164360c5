// Bluestein rows kept in one SM from the chirp-in to the chirp-out:
// M = Q 1024 points, Q = 5..24 (n = 2049 .. 12288), one CTA per row.
//
// The convolution needs no particular order of the spectrum, so the forward
// transform decimates in frequency and the inverse one in time, both in place
// in shared memory, with the spectrum in the digit-reversed order in between:
//   S1   x[m] w[m] (zero past n) from global memory; radix Q over points
//        j + 1024 r, times w_M^{j r}
//   S2   radix 32 over j2 + 32 s of each block of 1024, times w_1024^{j2 t}
//   S3   radix 32 over 32 neighbouring points: X[r + Q (t + 32 u)] at
//        1024 r + 32 t + u; times B there (stored in that order); radix 32 back
//   S2', S1'  the inverses; the first n points times scale w[m] to the output
// A point crosses shared memory eight times (8 bytes each), with one barrier
// per stage, and device memory once each way; M exceeds 2 n - 1 by at most 4095
// (between the built Q = 20 and 24; 2047 below), not by up to a factor of two.  n = 10007 (M = 20480), 2501 rows: 292 us,
// against 806 us for the two cluster-kernel passes over rows of 32768 points,
// whose exchange crosses SMs twice (n = 4099, 6000 rows: 299 against 868 us).
// What bounds it is the chain of stages with 16 warps per SM: issue slots 46 %
// used, shared memory about 30 %.  (One butterfly per thread in S2 and S3, 32 Q
// threads of 96 registers, measured no faster.)
//
// Slots: point m is at m ^ ((m / 32) & 15) (8-byte slots), so that the 32
// neighbouring points that a thread takes in S3 lie in other banks than its
// neighbours'; in S1 and S2 lanes take neighbouring points.
#include <complex>

#include "launch.h"
#include "plan.h"
#include "programmatic.h"

namespace fftseg {

namespace {

constexpr int kRow = 1024;  // the inner 32 x 32 points

template <int Q>
struct BlueRowShape {
    static constexpr int M = Q * kRow;
    // (Q = 24: 768 radix-32 butterflies in two full rounds, 286 -> 268 us at n = 12281)
    static constexpr int T = Q <= 6 ? 128 : Q <= 12 ? 256 : Q == 24 ? 384 : 512, PER_SM = 512 / T;
    static constexpr int A = (Q + 3) / 4;  // w_M^{j r}: r = 4 a + b, two factors
    static constexpr int H = Q / 2 + 1;    // points j + 1024 r < n have r < H (2 n - 1 <= M)
    static constexpr size_t SMEM = (size_t)(M + kRow) * sizeof(float2);
    static_assert(PER_SM * (SMEM + 1024) <= 228 * 1024, "rows per SM");
};

// The radix-Q butterfly.  Radix 10 and 20 as 2 x 5 and 4 x 5 with twiddles: half
// of S1's points are zero, whole inputs of their first butterflies, and they need
// fewer registers than the prime-factor form here (n = 10007: 291 against 311 us,
// n = 5003: 272 against 308).
template <int Q, int S>
FDEV void row_dft(float2 *v)
{
    if constexpr (Q == 10) dft_ab<2, 5, S>(v);
    else if constexpr (Q == 20) dft_ab<4, 5, S>(v);
    else dft<Q, S>(v);
}

template <int Q>
__global__ void __launch_bounds__(BlueRowShape<Q>::T, BlueRowShape<Q>::PER_SM) k_blue_row(const BlueRowArgs a)
{
    using Sh = BlueRowShape<Q>;
    constexpr int T = Sh::T, H = Sh::H, NB = 32 * Q;  // NB: radix-32 butterflies of a stage
    extern __shared__ float2 sm[];
    float2 *const TW = sm + Sh::M;  // w_1024^{j2 t} at [t][j2]
    const int tid = threadIdx.x;
    grid_launch_dependents();
    for (int e = tid; e < kRow; e += T) TW[e] = __ldg(a.tw2 + e);
    const int n = a.n;
    // w_M^{j r} from [b-1][j], b = 1..3, then [a-1][j] for w_M^{4 a j}
    auto tw1 = [&](int j, float2 (&w)[Q]) {
        float2 wb[4], wa[Sh::A];
#pragma unroll
        for (int b = 1; b < 4; ++b) wb[b] = __ldg(a.tw1 + (b - 1) * kRow + j);
#pragma unroll
        for (int i = 1; i < Sh::A; ++i) wa[i] = __ldg(a.tw1 + (2 + i) * kRow + j);
#pragma unroll
        for (int r = 1; r < Q; ++r) w[r] = r < 4 ? wb[r] : (r & 3) ? cmul(wa[r >> 2], wb[r & 3]) : wa[r >> 2];
    };
    grid_dependency_wait();
    __syncthreads();
    for (int64_t row = blockIdx.x; row < a.nseg; row += gridDim.x) {
        const float2 *const x = a.x + row * n;
        for (int j = tid; j < kRow; j += T) {  // S1
            // (every load before the first use: one after the other, each stage's
            // global loads cost a round trip per point, half of the row's time)
            float2 v[Q], w[Q], c[H];
#pragma unroll
            for (int r = 0; r < H; ++r) {
                v[r] = c[r] = make_float2(0.f, 0.f);
                if (j + kRow * r < n) {
                    v[r] = x[j + kRow * r];
                    c[r] = __ldg(a.w + j + kRow * r);
                }
            }
            tw1(j, w);
#pragma unroll
            for (int r = 0; r < H; ++r) v[r] = cmul(v[r], c[r]);
#pragma unroll
            for (int r = H; r < Q; ++r) v[r] = make_float2(0.f, 0.f);
            row_dft<Q, -1>(v);
            const int o = j ^ ((j >> 5) & 15);
            sm[o] = v[0];
#pragma unroll
            for (int r = 1; r < Q; ++r) sm[o + kRow * r] = cmul(v[r], w[r]);
        }
        __syncthreads();
        for (int b = tid; b < NB; b += T) {  // S2
            const int j2 = b & 31, o = (b >> 5) * kRow;
            float2 v[32];
#pragma unroll
            for (int s = 0; s < 32; ++s) v[s] = sm[o + 32 * s + (j2 ^ (s & 15))];
            dft<32, -1>(v);
            sm[o + j2] = v[0];
#pragma unroll
            for (int t0 = 0; t0 < 32; t0 += 8) {  // (twiddles in batches: a shared load stays behind a shared store)
                float2 w[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) w[i] = TW[32 * (t0 + i) + j2];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (t0 + i) sm[o + 32 * (t0 + i) + (j2 ^ ((t0 + i) & 15))] = cmul(v[t0 + i], w[i]);
            }
        }
        __syncthreads();
        for (int b = tid; b < NB; b += T) {  // S3: forward, times B, inverse
            const int o = b * 32, z = b & 15;
            float2 v[32], f[2][8];
#pragma unroll
            for (int i = 0; i < 8; ++i) f[0][i] = __ldg(a.bhat + i * NB + b);
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = sm[o + (q ^ z)];
            dft<32, -1>(v);
#pragma unroll
            for (int u = 0; u < 32; u += 8) {  // (B in batches, one ahead)
                if (u + 8 < 32) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) f[(u / 8 + 1) & 1][i] = __ldg(a.bhat + (u + 8 + i) * NB + b);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) v[u + i] = cmul(v[u + i], f[(u / 8) & 1][i]);
            }
            dft<32, 1>(v);
#pragma unroll
            for (int q = 0; q < 32; ++q) sm[o + (q ^ z)] = v[q];
        }
        // the next row on its way to L2
        if (tid == 0 && row + gridDim.x < a.nseg) {
            const uintptr_t p = reinterpret_cast<uintptr_t>(x + (int64_t)gridDim.x * n);
            const uintptr_t p0 = (p + 15) & ~(uintptr_t)15, p1 = (p + (uintptr_t)n * sizeof(float2)) & ~(uintptr_t)15;
            prefetch_l2_bulk(reinterpret_cast<const void *>(p0), (uint32_t)(p1 - p0));
        }
        __syncthreads();
        for (int b = tid; b < NB; b += T) {  // S2'
            const int j2 = b & 31, o = (b >> 5) * kRow;
            float2 v[32];
#pragma unroll
            for (int t = 0; t < 32; ++t) v[t] = sm[o + 32 * t + (j2 ^ (t & 15))];
#pragma unroll
            for (int t = 1; t < 32; ++t) v[t] = twmul<1>(v[t], TW[32 * t + j2]);
            dft<32, 1>(v);
#pragma unroll
            for (int s = 0; s < 32; ++s) sm[o + 32 * s + (j2 ^ (s & 15))] = v[s];
        }
        __syncthreads();
        for (int j = tid; j < kRow; j += T) {  // S1' (the same points as this thread's S1 of the next row)
            float2 v[Q], w[Q], c[H];
            tw1(j, w);
#pragma unroll
            for (int r = 0; r < H; ++r) {
                c[r] = make_float2(0.f, 0.f);
                if (j + kRow * r < n) c[r] = __ldg(a.w + j + kRow * r);
            }
            const int o = j ^ ((j >> 5) & 15);
            v[0] = sm[o];
#pragma unroll
            for (int r = 1; r < Q; ++r) v[r] = twmul<1>(sm[o + kRow * r], w[r]);
            row_dft<Q, 1>(v);
#pragma unroll
            for (int r = 0; r < H; ++r) {
                const int m = j + kRow * r;
                const float2 y = cscale(cmul(v[r], c[r]), a.scale);
                if (m < n) {
                    if (a.out_power) static_cast<float *>(a.out)[row * n + m] = y.x * y.x + y.y * y.y;
                    else static_cast<float2 *>(a.out)[row * n + m] = y;
                }
            }
        }
    }
}

template <int Q>
cudaError_t blue_row_t(const BlueRowArgs &a, cudaStream_t st)
{
    using Sh = BlueRowShape<Q>;
    auto k = k_blue_row<Q>;
    static int per_sm_dev[kMaxDevices] = {};  // per instantiation and device
    int &per_sm = per_sm_dev[current_device_slot()];
    if (per_sm == 0) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::SMEM);
        if (e != cudaSuccess) return e;
        int occ = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, Sh::T, Sh::SMEM);
        if (e != cudaSuccess) return e;
        if (occ < 1) return cudaErrorLaunchOutOfResources;
        per_sm = occ;
    }
    int64_t grid = (int64_t)per_sm * device_sm_count();
    if (grid > a.nseg) grid = a.nseg;
    if (grid < 1) return cudaSuccess;
    // a few rows: as k_one_sm (calls of 8 rows of 10007, one after the other: 20.7 ->
    // 18.0 us; the two cluster passes, which spread a row over eight SMs, 18.9)
    if (a.nseg <= device_sm_count() / 2) return launch_programmatic(k, (unsigned)grid, Sh::T, Sh::SMEM, st, a);
    k<<<(unsigned)grid, Sh::T, Sh::SMEM, st>>>(a);
    return cudaGetLastError();
}

using cd = std::complex<double>;

// The DFT of x[0], x[stride], ... (len points): halves while len is even, the
// direct sum for the odd rest; root: exp(-2 pi i m / M), m < M.
void host_dft(const cd *x, int64_t stride, int64_t len, cd *out, const std::vector<cd> &root)
{
    const int64_t M = (int64_t)root.size();
    if (len & 1) {
        for (int64_t k = 0; k < len; ++k) {
            cd s = 0;
            for (int64_t j = 0; j < len; ++j) s += x[j * stride] * root[(size_t)(j * k % len * (M / len))];
            out[k] = s;
        }
        return;
    }
    const int64_t h = len / 2;
    host_dft(x, 2 * stride, h, out, root);
    host_dft(x + stride, 2 * stride, h, out + h, root);
    for (int64_t k = 0; k < h; ++k) {
        const cd e = out[k], o = out[k + h] * root[(size_t)(k * (M / len))];
        out[k] = e + o;
        out[k + h] = e - o;
    }
}

}  // namespace

// The row length for n: the smallest built Q 1024 >= 2 n - 1, as Q; 0 if none.
int blue_row_q(int64_t n)
{
    for (int q : {5, 6, 7, 8, 9, 10, 12, 14, 15, 16, 18, 20, 24})
        if ((int64_t)q * kRow >= 2 * n - 1) return n > 2048 ? q : 0;
    return 0;
}

// The tables of a row kernel: tw2 (1024 entries), then tw1 ((2 + A) 1024), then
// B = DFT_M(b) in the kernel's order, b the conjugate chirp over M in double.
void blue_row_tables(int q, const std::vector<cd> &b, std::vector<float2> &h)
{
    const int64_t M = (int64_t)q * kRow;
    const int A = (q + 3) / 4;
    h.resize((size_t)(kRow + (2 + A) * kRow + M));
    for (int t = 0; t < 32; ++t) host_roots(h.data() + 32 * t, 32, kRow, t);
    float2 *t1 = h.data() + kRow;
    for (int i = 1; i < 4; ++i) host_roots(t1 + (i - 1) * kRow, kRow, M, i);
    for (int i = 1; i < A; ++i) host_roots(t1 + (2 + i) * kRow, kRow, M, 4 * i);
    std::vector<cd> root((size_t)M), B((size_t)M);
    for (int64_t m = 0; m < M; ++m) {
        const double ang = 6.283185307179586476925286766559 * (double)m / (double)M;
        root[(size_t)m] = cd(cos(ang), -sin(ang));
    }
    host_dft(b.data(), 1, M, B.data(), root);
    float2 *o = h.data() + kRow + (2 + A) * kRow;
    for (int64_t u = 0; u < 32; ++u)
        for (int64_t c = 0; c < 32 * q; ++c) {  // butterfly c = 32 r + t of S3, bin r + q (t + 32 u)
            const cd v = B[(size_t)(c / 32 + q * (c % 32 + 32 * u))];
            o[u * 32 * q + c] = make_float2((float)v.real(), (float)v.imag());
        }
}

cudaError_t launch_blue_row(int q, const float2 *tables, BlueRowArgs a, cudaStream_t st)
{
    a.tw2 = tables;
    a.tw1 = tables + kRow;
    a.bhat = a.tw1 + (2 + (q + 3) / 4) * kRow;
    switch (q) {
        case 5: return blue_row_t<5>(a, st);
        case 6: return blue_row_t<6>(a, st);
        case 7: return blue_row_t<7>(a, st);
        case 8: return blue_row_t<8>(a, st);
        case 9: return blue_row_t<9>(a, st);
        case 10: return blue_row_t<10>(a, st);
        case 12: return blue_row_t<12>(a, st);
        case 14: return blue_row_t<14>(a, st);
        case 15: return blue_row_t<15>(a, st);
        case 16: return blue_row_t<16>(a, st);
        case 18: return blue_row_t<18>(a, st);
        case 20: return blue_row_t<20>(a, st);
        case 24: return blue_row_t<24>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fftseg
