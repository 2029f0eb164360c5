// Real-signal segments (FFTSEG_FLAG_REAL): the split between a length-n real
// DFT and a length-M = n/2 complex DFT.
//
// Forward.  The n real samples of a segment, read as M complex values
// z[m] = x[2m] + i x[2m+1], go through the complex FFT: Z = DFT_M(z).  With
// A = Z[k], B = conj(Z[(M - k) mod M]) and w = w_n^k = exp(-2 pi i k / n):
//   Fe = (A + B) / 2        (the DFT of the even samples)
//   Fo = -i (A - B) / 2     (the DFT of the odd samples)
//   X[k]     = Fe + w Fo
//   X[M - k] = conj(Fe - w Fo)
// for k = 0 .. M/2, which gives the n/2 + 1 bins X[0..M] of the real DFT
// (X[0] and X[M] are real).  k_real_post does this per pair (k, M - k).
//
// Inverse.  From the bins X[0..M] (the imaginary parts of X[0] and X[M] are
// ignored, as for the real part of the Hermitian extension), with A = X[k],
// B = conj(X[M - k]):
//   Z[k] = (A + B) + i conj(w_n^k) (A - B)
// so that the inverse complex FFT of length M gives z[m] = x[2m] + i x[2m+1]
// with x[j] = sum over all n bins of the Hermitian extension times
// exp(+2 pi i j k / n) (unnormalised, the library's NORM_NONE).
// k_real_pre does this per pair (k, M - k).
//
// Both passes apply the real transform's scale.  The twiddle table holds the
// forward values w_n^k for k = 0 .. M/2, evaluated in double, rounded once.
#include "launch.h"
#include "programmatic.h"

namespace fftseg {

namespace {

constexpr int kRealThreads = 256;

FDEV float2 cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
FDEV float2 conjf2(float2 a) { return make_float2(a.x, -a.y); }
FDEV float2 scalef2(float2 a, float s) { return make_float2(a.x * s, a.y * s); }

// X[k] and X[M - k] (scaled) from Z[k], C = Z[(M - k) mod M] and w = w_n^k
FDEV void split_pair(float2 A, float2 C, float2 w, float scale, float2 &xk, float2 &xm)
{
    const float2 B = conjf2(C);
    const float2 fe = make_float2(0.5f * (A.x + B.x), 0.5f * (A.y + B.y));
    const float2 fo = make_float2(0.5f * (A.y - B.y), -0.5f * (A.x - B.x));  // -i (A - B) / 2
    const float2 wfo = cmul(w, fo);
    xk = scalef2(make_float2(fe.x + wfo.x, fe.y + wfo.y), scale);
    xm = scalef2(make_float2(fe.x - wfo.x, -(fe.y - wfo.y)), scale);  // conj(Fe - w Fo)
}

// Z[k] (scaled) from A = X[k], C = X[M - k] and v = conj(w_n^k):
// (A + conj(C)) + i v (A - conj(C)).  Z[M - k] is the same of (C, A, -w_n^k).
FDEV float2 join_bin(float2 A, float2 C, float2 v, float scale)
{
    const float2 B = conjf2(C);
    const float2 d = cmul(v, make_float2(A.x - B.x, A.y - B.y));
    return scalef2(make_float2(A.x + B.x - d.y, A.y + B.y + d.x), scale);
}

// One block covers kRealThreads pairs of one segment: block b -> segment
// b / bps, pairs (b % bps) * kRealThreads + threadIdx.x.
template <bool POWER>
__global__ void __launch_bounds__(kRealThreads) k_real_post(const RealArgs a)
{
    const int64_t bps = a.blocks_per_seg;
    const int64_t s = blockIdx.x / bps;
    const int k = (int)(blockIdx.x - s * bps) * kRealThreads + threadIdx.x;
    const int M = a.m;
    if (k > M / 2) return;
    const float2 *Z = a.zin + s * M;
    float2 xk, xm;
    split_pair(Z[k], Z[(M - k) & (M - 1)], __ldg(a.tw + k), a.scale, xk, xm);
    const int64_t o = s * (M + 1);
    if (POWER) {
        float *P = static_cast<float *>(a.out) + o;
        P[k] = xk.x * xk.x + xk.y * xk.y;
        if (2 * k != M) P[M - k] = xm.x * xm.x + xm.y * xm.y;
    } else {
        float2 *X = static_cast<float2 *>(a.out) + o;
        X[k] = xk;
        if (2 * k != M) X[M - k] = xm;
    }
}

__global__ void __launch_bounds__(kRealThreads) k_real_pre(const RealArgs a)
{
    const int64_t bps = a.blocks_per_seg;
    const int64_t s = blockIdx.x / bps;
    const int k = (int)(blockIdx.x - s * bps) * kRealThreads + threadIdx.x;
    const int M = a.m;
    if (k > M / 2) return;
    const float2 *X = a.xin + s * (M + 1);
    float2 A = X[k], C = X[M - k];
    if (k == 0) {  // the imaginary parts of the real bins X[0] and X[M] do not enter
        A.y = 0.f;
        C.y = 0.f;
    }
    const float2 w = __ldg(a.tw + k);  // w_n^k (forward value); conj(w) = exp(+2 pi i k / n)
    float2 *Z = static_cast<float2 *>(a.out) + s * M;
    Z[k] = join_bin(A, C, conjf2(w), a.scale);
    if (k != 0 && 2 * k != M) Z[M - k] = join_bin(C, A, make_float2(-w.x, -w.y), a.scale);
}

// Forward real segments of n = 2L <= 8192 points in one pass: the block
// kernel's persistent CTAs and bulk-copied tiles of whole segments (the L
// complex values of each), the L-point Stockham FFT, then the split above
// inside the tile: Z goes to the tile buffer in natural order and every
// thread forms bin pairs (k, L - k), written as n/2 + 1 bins.  Bound by memory
// and, up to n = 256, by the stores' partial lines: 2^29 samples of n = 256 ..
// 4096 take 673 .. 809 us, n = 8192 872 us (643 at the copy rate).  Eight pairs
// are read before the first is stored: one pair at a time, each waited for its
// shared-memory reads, 757 .. 906 and 1023 us.
template <int LOG_L>
__global__ void __launch_bounds__((BlockShape<LOG_L, kBlockLogE<LOG_L>>::T), (BlockShape<LOG_L, kBlockLogE<LOG_L>>::PER_SM))
    k_block_r2c(const RealBlockArgs a)
{
    using Sh = BlockShape<LOG_L, kBlockLogE<LOG_L>>;
    constexpr int L = 1 << LOG_L, W = 1 << Sh::LOG_W, E = Sh::E, T = Sh::T, V = E / T;
    extern __shared__ __align__(1024) float2 sm[];
    float2 *P = sm;
    float2 *X = sm + 2 * E;
    uint64_t *bar = reinterpret_cast<uint64_t *>(X + Sh::SLOTS);
    const int tid = threadIdx.x;
    if (smem_u32(P) & 127) {
        if (tid == 0) atomicOr(a.err, 2);
        return;
    }
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    auto tile_bytes = [&](int64_t u) {
        int64_t segs = a.nseg - u * W;
        if (segs > W) segs = W;
        return (uint32_t)(segs * L * (int64_t)sizeof(float2));
    };
    // (launched with programmatic stream serialization, as k_block: the L2
    // fetch of the first two tiles starts before the wait for the previous
    // kernel)
    grid_launch_dependents();
    if (tid == 0)
        for (int64_t u = blockIdx.x, q = 0; q < 2 && u < a.ntiles; ++q, u += gridDim.x)
            prefetch_l2_bulk(a.in + u * E, tile_bytes(u));
    grid_dependency_wait();
    auto issue = [&](int64_t u, int b) {
        if (tid == 0) {
            const uint32_t bytes = tile_bytes(u);
            fence_proxy_async();
            mbar_expect_tx(&bar[b], bytes);
            tma_load_1d(P + b * E, a.in + u * E, bytes, &bar[b]);
        }
    };
    int64_t u = blockIdx.x;
    if (u < a.ntiles) issue(u, 0);
    for (int k = 0; u < a.ntiles; u += gridDim.x, ++k) {
        const int b = k & 1;
        if (u + gridDim.x < a.ntiles) issue(u + gridDim.x, b ^ 1);
        mbar_wait(&bar[b], (k >> 1) & 1, a.err);
        float2 *Pb = P + b * E;
        float2 v[V];
        gather<LOG_L, Sh::LOG_W, false, T, 0>(v, [&](int c, int i) { return Pb[(c << LOG_L) + i]; });
        run_stages<LOG_L, Sh::LOG_W, false, -1, T, Sh::PS, 0, false>(v, X, a.twL);
        // Z of every segment of the tile, natural order, into the tile buffer
        // (its last reads were the gather, ordered by the stages' barriers)
        scatter_last<LOG_L, Sh::LOG_W, false, T>(v, [&](int c, int i, float2 x) { Pb[(c << LOG_L) + i] = x; });
        __syncthreads();
        const int64_t line0 = u * W;
        auto store = [&](int64_t o, float2 x) {
            if (a.out_power) static_cast<float *>(a.out)[o] = x.x * x.x + x.y * x.y;
            else static_cast<float2 *>(a.out)[o] = x;
        };
        if constexpr (LOG_L <= 4) {
            // pairs (kk, L - kk), kk = 0 .. L/2, one at a time (the batches below,
            // whose kk = 0 is a branch of its own, with a test of the output kind per
            // store: 2^26 samples of n = 8 145 us against 97, of 16 128 against 111)
            constexpr int PAIRS = L / 2 + 1;
            for (int p = tid; p < W * PAIRS; p += T) {
                const int c = p / PAIRS, kk = p - c * PAIRS;
                const int64_t seg = line0 + c;
                if (seg >= a.nseg) continue;
                float2 xk, xm;
                split_pair(Pb[(c << LOG_L) + kk], Pb[(c << LOG_L) + ((L - kk) & (L - 1))], __ldg(a.tw + kk), a.scale,
                           xk, xm);
                const int64_t o = seg * (L + 1);
                if (a.out_power) {
                    float *Q = static_cast<float *>(a.out) + o;
                    Q[kk] = xk.x * xk.x + xk.y * xk.y;
                    if (2 * kk != L) Q[L - kk] = xm.x * xm.x + xm.y * xm.y;
                } else {
                    float2 *Q = static_cast<float2 *>(a.out) + o;
                    Q[kk] = xk;
                    if (2 * kk != L) Q[L - kk] = xm;
                }
            }
        } else {
            // pairs (kk, L - kk), kk = 0 .. L/2 - 1; kk = 0 also does L/2.  A thread's
            // reads all come before its first store
            constexpr int NP = E / 2 / T;
            float2 A[NP], C[NP], w[NP];
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const int p = tid + q * T, c = p >> (LOG_L - 1), kk = p & (L / 2 - 1);
                A[q] = Pb[(c << LOG_L) + kk];
                C[q] = Pb[(c << LOG_L) + ((L - kk) & (L - 1))];
                w[q] = __ldg(a.tw + kk);
            }
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const int p = tid + q * T, c = p >> (LOG_L - 1), kk = p & (L / 2 - 1);
                const int64_t seg = line0 + c;
                if (seg >= a.nseg) continue;
                const int64_t o = seg * (L + 1);
                float2 xk, xm;
                split_pair(A[q], C[q], w[q], a.scale, xk, xm);
                store(o + kk, xk);
                store(o + L - kk, xm);
                if (kk == 0) {
                    const float2 m = Pb[(c << LOG_L) + L / 2];
                    split_pair(m, m, __ldg(a.tw + L / 2), a.scale, xk, xm);
                    store(o + L / 2, xk);
                }
            }
        }
        __syncthreads();  // P[b] and X read in full before they are reused
    }
}

// Inverse real segments of n = 2L <= 8192 points in one pass: tiles of whole
// segments' bins (L + 1 each, contiguous) arrive by bulk copies, the join above
// runs in place on the tile (each pair (k, L - k) belongs to one thread), then
// the L-point Stockham FFT, written as n samples.  A bulk copy must start and
// end on 16 bytes, and a segment has an odd number of 8-byte bins: a tile's
// copy is widened to 16-byte boundaries (one bin of a neighbouring segment at
// most), except at the end of the batch, where the last segment's bin X[L] is
// read from global memory instead.  Bound by memory: 2^29 samples of
// n = 256 .. 2048 take 678 .. 762 us, n = 8192 862 us (643 at the copy rate);
// a join pass before the transform, through a 512 MiB intermediate, moved each
// bin through memory twice more (1909 .. 1392, 1425 us; 2^23 samples of 1024:
// 37 us, now 22).
template <int LOG_L>
struct C2rShape : BlockShape<LOG_L, kBlockLogE<LOG_L>> {
    using B = BlockShape<LOG_L, kBlockLogE<LOG_L>>;
    static constexpr int BUF = (B::E + (1 << B::LOG_W) + 2 + 15) & ~15;  // bins per buffer, in whole 128 bytes
    static constexpr size_t SMEM = (size_t)(B::SLOTS + 2 * BUF) * sizeof(float2) + 2 * sizeof(uint64_t);
};

template <int LOG_L>
__global__ void __launch_bounds__((C2rShape<LOG_L>::T), (C2rShape<LOG_L>::PER_SM)) k_block_c2r(const RealBlockArgs a)
{
    using Sh = C2rShape<LOG_L>;
    constexpr int L = 1 << LOG_L, W = 1 << Sh::LOG_W, E = Sh::E, T = Sh::T, V = E / T, BUF = Sh::BUF;
    extern __shared__ __align__(1024) float2 sm[];
    float2 *P = sm;
    float2 *X = sm + 2 * BUF;
    uint64_t *bar = reinterpret_cast<uint64_t *>(X + Sh::SLOTS);
    const int tid = threadIdx.x;
    if (smem_u32(P) & 127) {
        if (tid == 0) atomicOr(a.err, 2);
        return;
    }
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    // tile u: bins [first, last) of the batch, copied from the even bin at or
    // before first to the even bin at or after last (before, at the batch's end)
    auto first_bin = [&](int64_t u) { return u * W * (int64_t)(L + 1); };
    auto copy_from = [&](int64_t u) { return first_bin(u) & ~(int64_t)1; };
    auto copy_bytes = [&](int64_t u) {
        const int64_t total = a.nseg * (int64_t)(L + 1);
        int64_t end = (first_bin(u + 1) + 1) & ~(int64_t)1;
        if (end > total) end = total & ~(int64_t)1;
        return (uint32_t)((end - copy_from(u)) * (int64_t)sizeof(float2));
    };
    grid_launch_dependents();
    if (tid == 0)
        for (int64_t u = blockIdx.x, q = 0; q < 2 && u < a.ntiles; ++q, u += gridDim.x)
            prefetch_l2_bulk(a.in + copy_from(u), copy_bytes(u));
    grid_dependency_wait();
    auto issue = [&](int64_t u, int b) {
        if (tid == 0) {
            const uint32_t bytes = copy_bytes(u);
            fence_proxy_async();
            mbar_expect_tx(&bar[b], bytes);
            tma_load_1d(P + b * BUF, a.in + copy_from(u), bytes, &bar[b]);
        }
    };
    int64_t u = blockIdx.x;
    if (u < a.ntiles) issue(u, 0);
    float *out = static_cast<float *>(a.out);
    for (int k = 0; u < a.ntiles; u += gridDim.x, ++k) {
        const int b = k & 1;
        if (u + gridDim.x < a.ntiles) issue(u + gridDim.x, b ^ 1);
        mbar_wait(&bar[b], (k >> 1) & 1, a.err);
        const int64_t line0 = u * W;
        float2 *Pb = P + b * BUF + (first_bin(u) & 1);
        // the join: pairs (kk, L - kk), kk = 0 .. L/2 - 1; kk = 0 also does L/2.
        // All reads of a thread come before its writes (segments past the
        // batch hold stale values, which are not stored)
        {
            constexpr int NP = E / 2 / T;
            float2 A[NP], C[NP], w[NP];
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const int p = tid + q * T, c = p >> (LOG_L - 1), kk = p & (L / 2 - 1);
                A[q] = Pb[c * (L + 1) + kk];
                C[q] = Pb[c * (L + 1) + L - kk];
                w[q] = __ldg(a.tw + kk);
            }
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const int p = tid + q * T, c = p >> (LOG_L - 1), kk = p & (L / 2 - 1);
                float2 *Z = Pb + c * (L + 1);
                if (kk == 0) {
                    if (line0 + c == a.nseg - 1) C[q] = __ldcg(a.in + a.nseg * (int64_t)(L + 1) - 1);
                    A[q].y = 0.f;  // the imaginary parts of the real bins X[0] and X[L] do not enter
                    C[q].y = 0.f;
                }
                const float2 z = join_bin(A[q], C[q], conjf2(w[q]), a.scale);
                const float2 m = kk == 0 ? join_bin(Z[L / 2], Z[L / 2], conjf2(__ldg(a.tw + L / 2)), a.scale)
                                         : join_bin(C[q], A[q], make_float2(-w[q].x, -w[q].y), a.scale);
                Z[kk] = z;
                Z[kk == 0 ? L / 2 : L - kk] = m;
            }
        }
        __syncthreads();
        float2 v[V];
        gather<LOG_L, Sh::LOG_W, false, T, 0>(v, [&](int c, int i) { return Pb[c * (L + 1) + i]; });
        run_stages<LOG_L, Sh::LOG_W, false, 1, T, Sh::PS, 0, false>(v, X, a.twL);
        scatter_last<LOG_L, Sh::LOG_W, false, T>(v, [&](int c, int i, float2 x) {
            if (line0 + c < a.nseg) reinterpret_cast<float2 *>(out)[(line0 + c) * L + i] = x;
        });
        __syncthreads();  // P[b] and X read in full before they are reused
    }
}

template <int LOG_L, bool INVERSE>
cudaError_t block_real_t(RealBlockArgs a, cudaStream_t st)
{
    using B = BlockShape<LOG_L, kBlockLogE<LOG_L>>;
    constexpr size_t SMEM = INVERSE ? C2rShape<LOG_L>::SMEM : B::SMEM;
    auto k = INVERSE ? k_block_c2r<LOG_L> : k_block_r2c<LOG_L>;
    static int per_sm_dev[kMaxDevices] = {};  // per instantiation and device
    int &per_sm = per_sm_dev[current_device_slot()];
    if (per_sm == 0) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
        if (e != cudaSuccess) return e;
        int occ = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, B::T, SMEM);
        if (e != cudaSuccess) return e;
        per_sm = occ > 0 ? occ : 1;
    }
    a.ntiles = (a.nseg + (1 << B::LOG_W) - 1) >> B::LOG_W;
    if (a.ntiles == 0) return cudaSuccess;
    int64_t grid = (int64_t)per_sm * device_sm_count();
    if (grid > a.ntiles) grid = a.ntiles;
    return launch_programmatic(k, (unsigned)grid, B::T, SMEM, st, a);
}

template <bool INVERSE>
cudaError_t block_real(int log_l, const RealBlockArgs &a, cudaStream_t st)
{
    switch (log_l) {
        case 1: return block_real_t<1, INVERSE>(a, st);
        case 2: return block_real_t<2, INVERSE>(a, st);
        case 3: return block_real_t<3, INVERSE>(a, st);
        case 4: return block_real_t<4, INVERSE>(a, st);
        case 5: return block_real_t<5, INVERSE>(a, st);
        case 6: return block_real_t<6, INVERSE>(a, st);
        case 7: return block_real_t<7, INVERSE>(a, st);
        case 8: return block_real_t<8, INVERSE>(a, st);
        case 9: return block_real_t<9, INVERSE>(a, st);
        case 10: return block_real_t<10, INVERSE>(a, st);
        case 11: return block_real_t<11, INVERSE>(a, st);
        case 12: return block_real_t<12, INVERSE>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_block_r2c(int log_l, const RealBlockArgs &a, cudaStream_t st) { return block_real<false>(log_l, a, st); }
cudaError_t launch_block_c2r(int log_l, const RealBlockArgs &a, cudaStream_t st) { return block_real<true>(log_l, a, st); }

cudaError_t launch_real(bool post, bool power, RealArgs a, int64_t nseg, cudaStream_t st)
{
    if (nseg <= 0) return cudaSuccess;
    a.blocks_per_seg = (a.m / 2 + 1 + kRealThreads - 1) / kRealThreads;
    const int64_t blocks = nseg * a.blocks_per_seg;
    if (blocks > 0x7fffffffll) return cudaErrorInvalidValue;
    if (post) {
        if (power) k_real_post<true><<<(unsigned)blocks, kRealThreads, 0, st>>>(a);
        else k_real_post<false><<<(unsigned)blocks, kRealThreads, 0, st>>>(a);
    } else {
        k_real_pre<<<(unsigned)blocks, kRealThreads, 0, st>>>(a);
    }
    return cudaGetLastError();
}

}  // namespace fftseg
