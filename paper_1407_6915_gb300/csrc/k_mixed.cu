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
// to the output: 200 -> 174 us for 40001 segments).  Among those it is the one,
// with its tile, that a model of the stages' bank conflicts and of the threads
// left idle finds fastest (mixed_cost below): a first stage of radix 16 stores
// at a stride of 16 points, all in one bank pair, so 1536 runs as 6 16 16 and
// not 16 16 6 (2^25 points: 142 us against 228).  (Stage outputs padded against
// the bank conflicts of the other stages, or the butterflies' slots from a
// table, measured no faster: the index arithmetic or the table's latency took
// what they gave.)
//
// Each CTA (persistent) takes tiles of floor(E / n) whole segments, E = 2048
// with 128 threads and four CTAs per SM (four barriers that do not wait for
// each other: 1000 points 174 -> 162 us), or 4096 with 256 threads and two
// where the segment is longer or fills the smaller tile badly (1029).  The next tile is copied in with one bulk copy while the current one runs its stages, ping-ponging
// between two shared buffers with one barrier per stage.  Stage twiddles are
// read through the read-only cache.
#include "engine.cuh"
#include "launch.h"
#include "programmatic.h"

namespace fftseg {

namespace {

constexpr int kMixEMax = 4096;  // the longest segment, and the larger tile
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
// power, to the output instead: consecutive threads, consecutive bins.  (A
// schedule of one stage has a whole segment in a thread: its bins go through
// the tile, or neighbouring threads would store n points apart.  2^25 points of
// n = 14: 192 us, through the tile 96; of n = 5 124 and 94.)
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
    // A tile arrives by one bulk copy issued by thread 0 and completed on an
    // mbarrier.  The copy must start and end on 16 bytes, two points: for odd n
    // it starts or ends up to one point outside the tile (which still fits the
    // buffer: a tile that is full has an even number of points), except at the
    // end of an odd batch, whose last point thread 0 reads by itself.
    __shared__ __align__(8) uint64_t bar[2];
    const int64_t total = a.nseg * (int64_t)n;
    auto copy_from = [&](int64_t t) { return (t * spt * (int64_t)n) & ~(int64_t)1; };
    auto copy_bytes = [&](int64_t t) {
        int64_t end = t * spt * (int64_t)n + count_of(t) * n;
        end = (end + 1) & ~(int64_t)1;
        if (end > total) end = total & ~(int64_t)1;
        return (uint32_t)((end - copy_from(t)) * (int64_t)sizeof(float2));
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
            prefetch_l2_bulk(a.in + copy_from(t), copy_bytes(t));
    grid_dependency_wait();
    uint32_t phase = 0;  // bit b: parity of the next completion of bar[b]
    auto load = [&](int64_t t, float2 *dst, int b) {
        if (threadIdx.x == 0) {
            const uint32_t bytes = copy_bytes(t);
            fence_proxy_async();  // this buffer's earlier generic accesses before the copy
            mbar_expect_tx(&bar[b], bytes);
            tma_load_1d(dst, a.in + copy_from(t), bytes, &bar[b]);
        }
    };
    int64_t t = blockIdx.x;
    if (t < a.ntiles) load(t, buf0, 0);
    int cur = 0;
    for (; t < a.ntiles; t += gridDim.x) {
        const int64_t tn = t + gridDim.x;
        if (tn < a.ntiles) load(tn, cur ? buf0 : buf1, cur ^ 1);
        mbar_wait(&bar[cur], (phase >> cur) & 1, a.err);
        phase ^= 1u << cur;
        const int64_t o0 = t * spt * (int64_t)n;
        float2 *src = (cur ? buf1 : buf0) + (o0 & 1), *dst = buf2;
        if (threadIdx.x == 0 && t == a.ntiles - 1 && (total & 1)) src[total - 1 - o0] = a.in[total - 1];
        __syncthreads();
        const int cnt = count_of(t);
        MixOut mo{nullptr, a.scale, a.out_power};
        for (int st = 0; st < a.nstages; ++st) {
            if (st == a.nstages - 1 && st > 0)
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
        if (a.nstages == 1) {  // (buf2 is next written after the next tile's first barrier)
            const int count = cnt * n;
            for (int e = threadIdx.x; e < count; e += T) {
                const float2 v = cscale(src[e], a.scale);
                if (a.out_power) static_cast<float *>(a.out)[o0 + e] = v.x * v.x + v.y * v.y;
                else static_cast<float2 *>(a.out)[o0 + e] = v;
            }
        }
        cur ^= 1;
    }
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

namespace {

// Wavefronts of a half-warp's 8-byte shared-memory access: the most of its
// different slots that share one of the 16 bank pairs.
int half_warp_wavefronts(const int *slot, int lanes)
{
    int count[16] = {}, most = 0;
    for (int i = 0; i < lanes; ++i) {
        bool again = false;
        for (int k = 0; k < i && !again; ++k) again = slot[k] == slot[i];
        if (again) continue;
        const int w = ++count[slot[i] & 15];
        if (w > most) most = w;
    }
    return most;
}

// Modelled time of a schedule, per point: what the kernel spends on a tile's
// stages, fitted to 26 lengths from 90 to 4050 (all within 14 %, us per 2^26
// points): 20 per butterfly point in the threads' passes, idle threads of a
// last pass included; 12.1 per wavefront of the stages' shared-memory accesses
// (in units of a half-warp), taken from the first four half-warps of a stage's
// butterflies; 379 per thread and stage for the barriers and the start.  (The
// constant 44 of the fit, the same for all, is left out.)  Tiles of 4096
// points take 7 % more at equal figures.
double stage_cost(int n, int R, int ns, bool last, int tile)
{
#ifdef FFTSEG_COUNT_STAGE_MODEL
    FFTSEG_COUNT_STAGE_MODEL;  // (a test counts them)
#endif
    const int T = tile / 16, cnt = tile / n, m = n / R, nb = cnt * m, passes = (nb + T - 1) / T;
    int wave = 0, lanes = 0;
    for (int g0 = 0; g0 < 64 && g0 < nb; g0 += 16) {
        int in[16], out[16], k = 0;
        for (; k < 16 && g0 + k < nb; ++k) {
            const int g = g0 + k, j = g % m, base = g / m * n;
            in[k] = base + j;
            out[k] = base + j / ns * ns * R + j % ns;
        }
        wave += half_warp_wavefronts(in, k);
        if (!last) wave += half_warp_wavefronts(out, k);  // (the last stage stores to the output)
        lanes += k;
    }
    return 20.0 * passes * R * T + 12.1 * 16.0 * wave / lanes * R * nb + 379.0 * T;
}

struct MixedBest {
    double cost;
    int tile, radix[kMixMaxStages];
    // a stage's cost depends on its radix and ns alone (and on being the last, and
    // the tile): kept by a hash of these, modelled about once each (every schedule
    // by itself took up to 2.9 ms of a plan's creation, n = 4032, now 0.3)
    int key[1024];
    double stage[1024];
};

double mixed_cost(int n, const int *radix, int nstages, int tile, MixedBest &best)
{
    double c = 0;
    for (int t = 0, ns = 1; t < nstages; ns *= radix[t++]) {
        const bool last = t == nstages - 1;
        const int key = ((ns * 32 + radix[t]) * 2 + last) * 2 + (tile == kMixEMax), i = (int)((unsigned)key * 2654435769u >> 22);
        if (best.key[i] != key) {
            best.key[i] = key;
            best.stage[i] = stage_cost(n, radix[t], ns, last, tile);
        }
        c += best.stage[i];
    }
    return c / (tile / n * (double)n) * (tile == kMixEMax ? 1.07 : 1.0);
}

// All orders of all factorisations of m into `left` radices, after `depth` of them.
void mixed_search(int n, int m, int left, int *radix, int depth, MixedBest &best)
{
    if (left == 0) {
        if (m != 1) return;
        for (int tile = 2048; tile <= kMixEMax; tile *= 2) {
            if (n > tile) continue;
            const double c = mixed_cost(n, radix, depth, tile, best);
            if (best.cost > 0 && c >= best.cost) continue;
            best.cost = c;
            best.tile = tile;
            for (int i = 0; i < depth; ++i) best.radix[i] = radix[i];
        }
        return;
    }
    for (int r : {16, 15, 14, 12, 10, 9, 8, 7, 6, 5, 4, 3, 2}) {
        if (m % r || m > r << 4 * (left - 1)) continue;
        radix[depth] = r;
        mixed_search(n, m / r, left - 1, radix, depth + 1, best);
    }
}

}  // namespace

// The schedule of the fewest stages, and the tile, of the least modelled time.
bool mixed_schedule(int64_t n, int *nstages, int *radix, int *tile)
{
    if (n < 2 || n > kMixEMax) return false;
    int64_t m = n;
    for (int p : {7, 5, 3, 2})
        while (m % p == 0) m /= p;
    if (m != 1) return false;
    for (int s = 1; s <= kMixMaxStages; ++s) {
        MixedBest best{};
        mixed_search((int)n, (int)n, s, radix, 0, best);
        if (best.cost == 0) continue;
        for (int i = 0; i < s; ++i) radix[i] = best.radix[i];
        *nstages = s;
        *tile = best.tile;
        return true;
    }
    return false;
}

cudaError_t launch_mixed(int sign, const MixedArgs &a, cudaStream_t st)
{
    if (a.tile == 2048) return sign < 0 ? mixed_t<-1, 2048>(a, st) : mixed_t<1, 2048>(a, st);
    return sign < 0 ? mixed_t<-1, 4096>(a, st) : mixed_t<1, 4096>(a, st);
}

}  // namespace fftseg
