// Lengths n = 2^a 3^b 5^c 7^d <= 4096 that are not powers of two, in one
// pass: mixed-radix Stockham stages of radix 2..10, 12, 14, 15 or 16.
//
// The Cooley-Tukey factorisation (Sec. I of the paper) holds for any
// factorisation n = R_1 R_2 ... R_s; the FFT libraries the paper names handle
// such lengths natively.  Stage t (radix R, Ns = R_1 ... R_{t-1} points
// already combined) runs the n/R butterflies j of every segment:
//   a_r = line[j + r n/R], times w_{Ns R}^{(j mod Ns) r} (r >= 1),
//   A = DFT_R(a),  line'[(j / Ns) Ns R + (j mod Ns) + r Ns] = A_r,
// the self-sorting Stockham form, so the bins come out in natural order.
// The schedule has as few stages as the length allows: every stage is one
// write and one read of the tile in shared memory and a barrier, which is what
// the kernel spends its time on (1000 = 10 10 10 in three stages instead of
// 5 5 5 8 in four, with the last stage's bins going from registers straight
// to the output: 200 -> 174 us for 40001 segments).  Odd radices come first:
// their Ns = 1 stage stores with an odd stride, which no two lanes of a
// half-warp share a bank pair with.  (Stage outputs padded against the bank
// conflicts of the other stages, or the butterflies' slots from a table,
// measured no faster: the index arithmetic or the table's latency took what
// they gave.)
//
// Each CTA (persistent) takes tiles of floor(E / n) whole segments, E = 2048
// with 128 threads and four CTAs per SM up to n = 2048 (four barriers that do
// not wait for each other: 1000 points 174 -> 162 us), else 4096 with 256
// threads and two.  The next tile is copied in with one bulk copy (or 8-byte cp.async
// copies by every thread) while the current one runs its stages, ping-ponging
// between two shared buffers with one barrier per stage.  Stage twiddles are
// read through the read-only cache.
#include "engine.cuh"
#include "launch.h"
#include "programmatic.h"

namespace fftseg {

namespace {

constexpr int kMixEMax = 4096;  // the longest segment
int mix_tile(int64_t n) { return n <= 2048 ? 2048 : 4096; }  // points per tile buffer
template <int E>
constexpr int kMixThreads = E / 16;

// x / d for 0 <= x < 2^20 and a runtime divisor d with rd ~ 1/d: the float
// quotient is within one of the true one, then one correction step.
FDEV int divq(int x, int d, float rd)
{
    int q = __float2int_rz((float)x * rd);
    const int r = x - q * d;
    if (r < 0) --q;
    else if (r >= d) ++q;
    return q;
}

// One stage of a tile of cnt segments.  The last stage (out not null: ns =
// n / R, butterfly j gives bins j + r ns) scales and stores its bins, or their
// power, to the output instead: consecutive threads, consecutive bins.
struct MixOut {
    void *out;  // this tile's first bin, or null
    float scale;
    int power;
};

template <int R, int S, int T>
FDEV void mix_stage(const float2 *src, float2 *dst, int cnt, int n, int ns, float rm, float rns,
                    const float2 *__restrict__ tw, const MixOut &mo, [[maybe_unused]] int *err)
{
    const int m = n / R;
    const int nb = cnt * m;
    // butterfly g = seg m + j, stepped by T without a division per step
    int seg = divq(threadIdx.x, m, rm);
    int j = threadIdx.x - seg * m;
    const int dseg = divq(T, m, rm), dj = T - dseg * m;
    for (int g = threadIdx.x; g < nb; g += T) {
        const int base = seg * n;
        float2 x[R];
        // (self-checking build: the butterfly's points lie in the tile)
        const bool ok = FFTSEG_CHECK(seg < cnt && j < m && base + n <= cnt * n, err);
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = ok ? src[base + j + r * m] : make_float2(0.f, 0.f);
        int jq = j, k = 0;
        if (ns > 1) {
            jq = divq(j, ns, rns);
            k = j - jq * ns;
#pragma unroll
            for (int r = 1; r < R; ++r) x[r] = twmul<S>(x[r], __ldg(tw + (r - 1) * ns + k));
        }
        dft<R, S>(x);
        const int o = base + jq * ns * R + k;
        if (FFTSEG_CHECK(o + (R - 1) * ns < base + n && k < ns, err)) {
            if (!mo.out) {
#pragma unroll
                for (int r = 0; r < R; ++r) dst[o + r * ns] = x[r];
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float2 v = cscale(x[r], mo.scale);
                    if (mo.power) static_cast<float *>(mo.out)[o + r * ns] = v.x * v.x + v.y * v.y;
                    else static_cast<float2 *>(mo.out)[o + r * ns] = v;
                }
            }
        }
        seg += dseg;
        j += dj;
        if (j >= m) {
            j -= m;
            ++seg;
        }
    }
}

template <int S, int E>
__global__ void __launch_bounds__(kMixThreads<E>, 8192 / E) k_mixed(const __grid_constant__ MixedArgs a)
{
    extern __shared__ __align__(16) float2 smx[];
    constexpr int T = kMixThreads<E>;
    float2 *const buf0 = smx, *const buf1 = smx + E, *const buf2 = smx + 2 * E;
    const int n = a.n, spt = a.segs_per_tile;
    auto count_of = [&](int64_t t) -> int {
        const int64_t left = a.nseg - t * spt;
        return (int)(left < spt ? left : spt);
    };
    // A tile whose bytes start on a 16-byte boundary and are a multiple of 16
    // (an even number of points) arrives by one bulk copy issued by thread 0
    // and completed on an mbarrier; otherwise every thread issues 8-byte
    // cp.async copies.
    __shared__ __align__(8) uint64_t bar[2];
    auto bulk_ok = [&](int64_t t) -> bool {
        return ((t * spt * (int64_t)n) & 1) == 0 && ((count_of(t) * n) & 1) == 0;
    };
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    // (launched with programmatic stream serialization, as k_block: the L2
    // fetch of the first two bulk-copied tiles starts before the wait for the
    // previous kernel)
    grid_launch_dependents();
    if (threadIdx.x == 0)
        for (int64_t t = blockIdx.x, q = 0; q < 2 && t < a.ntiles; ++q, t += gridDim.x)
            if (bulk_ok(t))
                prefetch_l2_bulk(a.in + t * spt * (int64_t)n, (uint32_t)(count_of(t) * n * sizeof(float2)));
    grid_dependency_wait();
    uint32_t phase = 0;  // bit b: parity of the next completion of bar[b]
    auto load = [&](int64_t t, float2 *dst, int b) {
        const float2 *src = a.in + t * spt * (int64_t)n;
        const int count = count_of(t) * n;
        if (bulk_ok(t)) {
            if (threadIdx.x == 0) {
                fence_proxy_async();  // this buffer's earlier generic accesses before the copy
                mbar_expect_tx(&bar[b], (uint32_t)(count * sizeof(float2)));
                tma_load_1d(dst, src, (uint32_t)(count * sizeof(float2)), &bar[b]);
            }
        } else {
            for (int e = threadIdx.x; e < count; e += T) cp_async8(dst + e, src + e, 8);
        }
    };
    int64_t t = blockIdx.x;
    if (t < a.ntiles) load(t, buf0, 0);
    cp_async_commit();
    int cur = 0;
    for (; t < a.ntiles; t += gridDim.x) {
        const int64_t tn = t + gridDim.x;
        if (tn < a.ntiles) load(tn, cur ? buf0 : buf1, cur ^ 1);
        cp_async_commit();
        cp_async_wait<1>();  // this tile's copies (the group before the one just issued)
        if (bulk_ok(t)) {
            mbar_wait(&bar[cur], (phase >> cur) & 1, a.err);
            phase ^= 1u << cur;
        }
        __syncthreads();
        const int cnt = count_of(t);
        float2 *src = cur ? buf1 : buf0, *dst = buf2;
        const int64_t o0 = t * spt * (int64_t)n;
        MixOut mo{nullptr, a.scale, a.out_power};
        for (int st = 0; st < a.nstages; ++st) {
            if (st == a.nstages - 1)
                mo.out = a.out_power ? (void *)(static_cast<float *>(a.out) + o0)
                                     : (void *)(static_cast<float2 *>(a.out) + o0);
            const float2 *tw = a.tw + a.twoff[st];
            const int ns = a.ns[st];
            const float rm = a.rm[st], rns = a.rns[st];
            switch (a.radix[st]) {
                case 2: mix_stage<2, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 3: mix_stage<3, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 4: mix_stage<4, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 5: mix_stage<5, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 6: mix_stage<6, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 7: mix_stage<7, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 8: mix_stage<8, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 9: mix_stage<9, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 10: mix_stage<10, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 12: mix_stage<12, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 14: mix_stage<14, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                case 15: mix_stage<15, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
                default: mix_stage<16, S, T>(src, dst, cnt, n, ns, rm, rns, tw, mo, a.err); break;
            }
            __syncthreads();  // (after the last stage: its buffer may be refilled)
            float2 *tmp = src;
            src = dst;
            dst = tmp;
        }
        cur ^= 1;
    }
    cp_async_wait<0>();
}

template <int S, int E>
cudaError_t mixed_t(const MixedArgs &a, cudaStream_t st)
{
    auto k = k_mixed<S, E>;
    constexpr size_t SMEM = 3 * E * sizeof(float2);
    constexpr int T = kMixThreads<E>;
    static int per_sm_dev[kMaxDevices] = {};  // per instantiation and device
    int &per_sm = per_sm_dev[current_device_slot()];
    if (per_sm == 0) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
        if (e != cudaSuccess) return e;
        int occ = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, T, SMEM);
        if (e != cudaSuccess) return e;
        if (occ < 1) return cudaErrorLaunchOutOfResources;
        per_sm = occ;
    }
    if (a.ntiles == 0) return cudaSuccess;
    int64_t grid = (int64_t)per_sm * device_sm_count();
    if (grid > a.ntiles) grid = a.ntiles;
    return launch_programmatic(k, (unsigned)grid, T, SMEM, st, a);
}

}  // namespace

int mixed_segments_per_tile(int64_t n) { return n <= kMixEMax ? (int)(mix_tile(n) / n) : 0; }

namespace {

// The fewest stages whose radices multiply to m, each at most `top`; among
// those the smallest largest radix.  Radices come out in falling order.
bool mixed_search(int64_t m, int top, int left, int *radix, int depth)
{
    static const int R[] = {16, 15, 14, 12, 10, 9, 8, 7, 6, 5, 4, 3, 2};
    if (left == 0) return m == 1;
    for (int r : R) {
        if (r > top || m % r) continue;
        radix[depth] = r;
        if (mixed_search(m / r, r, left - 1, radix, depth + 1)) return true;
    }
    return false;
}

}  // namespace

bool mixed_schedule(int64_t n, int *nstages, int *radix)
{
    if (n < 2 || n > kMixEMax) return false;
    int64_t m = n;
    for (int p : {7, 5, 3, 2})
        while (m % p == 0) m /= p;
    if (m != 1) return false;
    for (int s = 1; s <= kMixMaxStages; ++s)
        for (int top = 2; top <= 16; ++top)
            if (mixed_search(n, top, s, radix, 0)) {
                // odd radices first
                for (int i = 1; i < s; ++i)
                    for (int j = i; j > 0 && (radix[j] & 1) > (radix[j - 1] & 1); --j) {
                        const int t = radix[j];
                        radix[j] = radix[j - 1];
                        radix[j - 1] = t;
                    }
                *nstages = s;
                return true;
            }
    return false;
}

cudaError_t launch_mixed(int sign, const MixedArgs &a, cudaStream_t st)
{
    if (mix_tile(a.n) == 2048) return sign < 0 ? mixed_t<-1, 2048>(a, st) : mixed_t<1, 2048>(a, st);
    return sign < 0 ? mixed_t<-1, 4096>(a, st) : mixed_t<1, 4096>(a, st);
}

}  // namespace fftseg
