// Instantiations and launchers of k_lines: the single-pass block kernel
// (n <= 4096) and the column/row passes of the two-pass path.
#include "launch.h"
#include "programmatic.h"

namespace fftseg {

namespace {

int g_sm_count[kMaxDevices] = {};

int sm_count()
{
    int &c = g_sm_count[current_device_slot()];
    if (c == 0) {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        c = v > 0 ? v : 1;
    }
    return c;
}

template <int LOG_L, int S, int PREC = PREC_FP32, int LOG_E = 12>
cudaError_t block_t(BlockArgs a, cudaStream_t st)
{
    // Up to 2^22 points (32 MiB) in tiles of 2048 points: a launch is at most a few
    // rounds of the grid then (as many with either tile, the CTAs per SM double
    // with the tiles), and tiles half as large are in sooner and out sooner, at
    // the start and the end.  Replayed from a graph over rotating buffers, us with
    // tiles of 4096 -> 2048 points: n = 1024, 2^18 points 3.63 -> 2.98, 2^20 5.12 ->
    // 4.61, 2^22 13.53 -> 12.83; n = 32 3.94 -> 3.21, 5.60 -> 5.29, 15.4 -> 14.9;
    // n = 2048 3.63 -> 2.97, 5.17 -> 4.78, 14.1 -> 13.3; the lengths between and
    // |X|^2 alike.  From 2^23 points on equal, above up to 5 % slower.  The same
    // arithmetic on every segment, so the same bits.
    if constexpr (PREC == PREC_FP32 && LOG_E == 12 && kBlockLogE<LOG_L> == 11) {
        if (a.nseg <= (int64_t(1) << 22) >> LOG_L) return block_t<LOG_L, S, PREC, 11>(a, st);
    }
    using B = BlockShape<LOG_L, LOG_E>;
    auto k = k_block<LOG_L, S, PREC, LOG_E>;
    a.ntiles = (a.nseg + (1 << B::LOG_W) - 1) >> B::LOG_W;
    static int per_sm_dev[kMaxDevices] = {};  // per instantiation and device
    int &per_sm = per_sm_dev[current_device_slot()];
    if (per_sm == 0) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)B::SMEM);
        if (e != cudaSuccess) return e;
        int occ = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, B::T, B::SMEM);
        if (e != cudaSuccess) return e;
        per_sm = occ > 0 ? occ : 1;
    }
    if (a.ntiles == 0) return cudaSuccess;
    int64_t grid = (int64_t)per_sm * sm_count();
    if (grid > a.ntiles) grid = a.ntiles;
    // the blocks of back-to-back batches take the SMs as the previous grid
    // leaves them (the kernel waits for the previous kernel's writes before it
    // touches global memory)
    return launch_programmatic(k, (unsigned)grid, B::T, B::SMEM, st, a);
}

// Segments of n = 4, 8 and 16 points: a warp takes 512 points, 16 (whole
// segments) a lane, and needs no barrier but its own.  The points come in by
// coalesced 16-byte loads and change to 16 a lane through the warp's own 4 KiB;
// the bins go back the same way.  Row l (lane l's points) holds 16-byte chunk c
// at c ^ (l mod 8), |X|^2 rows (64 bytes) at c ^ (l / 2 mod 4): conflict-free on
// both sides.  Bound by memory: 2^26 points take 180 us (0.89 of the copy rate),
// as |X|^2 132 us.  (On the tiles of k_block a thread read its points at a stride
// of a segment, 32 lanes of n = 16 in one bank pair, and stored them so: n = 16
// 430 us, |X|^2 327; n = 8 310; n = 4 255.  n = 4 as |X|^2 stays there, see
// launch_block, and n = 2: 176 us against
// 182, |X|^2 122 against 134.)
constexpr int kShortWarps = 8;

template <int LOG_L, int S>
__global__ void __launch_bounds__(32 * kShortWarps, 4) k_short(const BlockArgs a)
{
    constexpr int L = 1 << LOG_L;
    static_assert(LOG_L >= 2 && LOG_L <= 4, "whole segments in 16 points");
    __shared__ float4 sm[kShortWarps * 256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    float4 *const X = sm + warp * 256;
    const int64_t total = a.nseg << LOG_L;
    grid_launch_dependents();
    grid_dependency_wait();
    for (int64_t u = (int64_t)blockIdx.x * warps + warp; u * 512 < total; u += (int64_t)gridDim.x * warps) {
        const int left = (int)(total - u * 512 < 512 ? total - u * 512 : 512);  // points, a multiple of 4
        const float4 *const in = reinterpret_cast<const float4 *>(a.in + u * 512);
        float4 q[8];
#pragma unroll
        for (int r = 0; r < 8; ++r)
            q[r] = 2 * (32 * r + lane) < left ? in[32 * r + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
        __syncwarp();  // the unit before has been read
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int row = 4 * r + (lane >> 3);
            X[8 * row + ((lane ^ row) & 7)] = q[r];
        }
        __syncwarp();
        float2 v[16];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float4 x = X[8 * lane + (c ^ (lane & 7))];
            v[2 * c] = make_float2(x.x, x.y);
            v[2 * c + 1] = make_float2(x.z, x.w);
        }
#pragma unroll
        for (int g = 0; g < 16; g += L) dft<L, S>(v + g);
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = cscale(v[c], a.scale);
        if (a.out_power) {
            __syncwarp();  // (rows change size)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                X[4 * lane + (c ^ ((lane >> 1) & 3))] = make_float4(power_of(v[4 * c]), power_of(v[4 * c + 1]),
                                                                    power_of(v[4 * c + 2]), power_of(v[4 * c + 3]));
            __syncwarp();
            float *const out = static_cast<float *>(a.out) + u * 512;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int row = 8 * r + (lane >> 2), e = 4 * (32 * r + lane);
                const float4 x = X[4 * row + ((lane ^ (row >> 1)) & 3)];
                if (e < left) *reinterpret_cast<float4 *>(out + e) = x;
            }
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c)  // (this lane's own row)
                X[8 * lane + (c ^ (lane & 7))] = make_float4(v[2 * c].x, v[2 * c].y, v[2 * c + 1].x, v[2 * c + 1].y);
            __syncwarp();
            float4 *const out = reinterpret_cast<float4 *>(static_cast<float2 *>(a.out) + u * 512);
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int row = 4 * r + (lane >> 3);
                const float4 x = X[8 * row + ((lane ^ row) & 7)];
                if (2 * (32 * r + lane) < left) out[32 * r + lane] = x;
            }
        }
    }
}

template <int LOG_L, int S>
cudaError_t short_t(const BlockArgs &a, cudaStream_t st)
{
    auto k = k_short<LOG_L, S>;
    static int per_sm_dev[kMaxDevices] = {};  // per instantiation and device
    int &per_sm = per_sm_dev[current_device_slot()];
    if (per_sm == 0) {
        int occ = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, 32 * kShortWarps, 0);
        if (e != cudaSuccess) return e;
        per_sm = occ > 0 ? occ : 1;
    }
    // A small batch is spread over the SMs, in smaller CTAs (2^14 points of n = 4,
    // 32 warps: in 4 CTAs 2.07 us, in 32 1.37, on the tiles of k_block 1.48)
    const int64_t units = ((a.nseg << LOG_L) + 511) / 512;
    if (units == 0) return cudaSuccess;
    int64_t warps = (units + sm_count() - 1) / sm_count();
    if (warps > kShortWarps) warps = kShortWarps;
    const int64_t ctas = (units + warps - 1) / warps;
    int64_t grid = (int64_t)per_sm * sm_count();
    if (grid > ctas) grid = ctas;
    return launch_programmatic(k, (unsigned)grid, 32 * (unsigned)warps, 0, st, a);
}

template <int LOG_L>
struct PassShape {
    // up to 16 lines of up to 1024 points (16 KB..128 KB per tile)
    static constexpr int LOG_W = (14 - LOG_L) < 4 ? (14 - LOG_L) : 4;
    static constexpr int T = (1 << (LOG_L + LOG_W)) / 16;
    static constexpr int SLOTS = smem_slots<LOG_L, LOG_W, 4>();
};

template <int LOG_L, int S>
cudaError_t pass_t(const LinesArgs &a, int64_t units, cudaStream_t st)
{
    using P = PassShape<LOG_L>;
    auto k = k_lines<LOG_L, P::LOG_W, true, S, P::T>;
    const size_t smem = (size_t)P::SLOTS * sizeof(float2);
    static bool configured_dev[kMaxDevices] = {};  // per instantiation and device
    bool &configured = configured_dev[current_device_slot()];
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    if (units == 0) return cudaSuccess;
    k<<<(unsigned)units, P::T, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

int device_sm_count() { return sm_count(); }

int pass_log_w(int log_l)
{
    return (14 - log_l) < 4 ? (14 - log_l) : 4;
}

#define FFTSEG_BLOCK_CASE(LL) \
    case LL: return sign < 0 ? block_t<LL, -1>(a, st) : block_t<LL, 1>(a, st);

#define FFTSEG_SHORT_CASE(LL) \
    case LL: return sign < 0 ? short_t<LL, -1>(a, st) : short_t<LL, 1>(a, st);

cudaError_t launch_block(int log_n, int sign, int prec, const BlockArgs &a, cudaStream_t st)
{
    if (prec != PREC_FP32) {  // tensor-core radix-16 stages: n a power of 16
#define FFTSEG_BLOCK_TC(LL)                                                                                   \
    case LL:                                                                                                  \
        if (prec == PREC_FP16) return sign < 0 ? block_t<LL, -1, PREC_FP16>(a, st) : block_t<LL, 1, PREC_FP16>(a, st); \
        return sign < 0 ? block_t<LL, -1, PREC_BF16>(a, st) : block_t<LL, 1, PREC_BF16>(a, st);
        switch (log_n) {
            FFTSEG_BLOCK_TC(4)
            FFTSEG_BLOCK_TC(8)
            FFTSEG_BLOCK_TC(12)
            default: return cudaErrorInvalidValue;
        }
    }
    switch (log_n) {
        FFTSEG_BLOCK_CASE(1)
        case 2:  // |X|^2: 2^20 points 2.7 us on the tiles, 3.7 a warp at a time (2^25: 63 and 65)
            if (a.out_power) return sign < 0 ? block_t<2, -1>(a, st) : block_t<2, 1>(a, st);
            return sign < 0 ? short_t<2, -1>(a, st) : short_t<2, 1>(a, st);
        FFTSEG_SHORT_CASE(3)
        FFTSEG_SHORT_CASE(4)
        FFTSEG_BLOCK_CASE(5)
        FFTSEG_BLOCK_CASE(6)
        FFTSEG_BLOCK_CASE(7)
        FFTSEG_BLOCK_CASE(8)
        FFTSEG_BLOCK_CASE(9)
        FFTSEG_BLOCK_CASE(10)
        FFTSEG_BLOCK_CASE(11)
        FFTSEG_BLOCK_CASE(12)
        default: return cudaErrorInvalidValue;
    }
}

#define FFTSEG_PASS_CASE(LL) \
    case LL: return sign < 0 ? pass_t<LL, -1>(a, units, st) : pass_t<LL, 1>(a, units, st);

cudaError_t launch_pass(int log_l, int sign, const LinesArgs &a, int64_t units, cudaStream_t st)
{
    switch (log_l) {
        FFTSEG_PASS_CASE(4)
        FFTSEG_PASS_CASE(5)
        FFTSEG_PASS_CASE(6)
        FFTSEG_PASS_CASE(7)
        FFTSEG_PASS_CASE(8)
        FFTSEG_PASS_CASE(9)
        FFTSEG_PASS_CASE(10)
        FFTSEG_PASS_CASE(11)
        FFTSEG_PASS_CASE(12)
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fftseg
