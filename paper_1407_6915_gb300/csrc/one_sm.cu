// Segments of n = 2^14 points in one SM each: the whole segment (128 KiB) in
// shared memory, one CTA of 512 threads with 32 points each.
//
// Decimation in frequency, in place: index m = (a, b, c), a, b < 32, c < 16
// (m = 512 a + 16 b + c).
//   S1  radix 32 over a from global memory, times w_n^{j k_a}, j = m mod 512
//   S2  radix 32 over b, times w_512^{c k_b}
//   S3  radix 16 over c: X[k_a + 32 k_b + 1024 k_c], to global memory
// Three barriers and 43 bytes of shared-memory traffic per point (two exchanges,
// and the rows copied ahead), and no traffic between SMs.  4001 segments: 181 us (0.87 of the copy rate), against 252 us (0.62)
// for the 4-CTA cluster kernel, which waits for its all-to-all exchange between
// SMs.  22 of the next segment's 32 rows are copied into the shared memory left
// over while a segment runs (199 us with all of them read when it starts).  (Four
// stages of radix 16, 16, 16, 4 with 1024 threads of 64 registers
// measured 266 us: half as much shared-memory traffic again and a barrier more,
// and with one CTA per SM nothing overlaps a stage.)  2^15 does not fit an SM; at
// 2^13 the 2-CTA cluster kernel runs at 0.61 of the copy rate (2000 segments 64
// us), and this form has not been tried there.
//
// Slot of m: m ^ (a mod 16) (8-byte slots).  In S1 and S2 a half-warp takes 16
// neighbouring m; in S3 16 neighbouring a of one (b, c), so that a warp stores 32
// neighbouring bins.  All conflict-free.
#include "launch.h"
#include "plan.h"
#include "programmatic.h"

namespace fftseg {

namespace {

constexpr int kN = 1 << 14, kT = 512;
constexpr int kTw2 = 10 * 512, kTw = kTw2 + 31 * 16;  // w_n^{j r} factors, then w_512^{c r}
constexpr int kAhead = 22;  // rows of 512 points of the next segment copied in while this one runs
constexpr size_t kSmem = (size_t)(kN + 31 * 16 + kAhead * 512) * sizeof(float2) + sizeof(uint64_t);

template <int S>
__global__ void __launch_bounds__(kT, 1) k_one_sm(const OneSmArgs a)
{
    extern __shared__ float2 sm[];
    const int tid = threadIdx.x;
    float2 *const P = sm + kN;              // rows ahead
    float2 *const T2 = P + kAhead * 512;    // [r-1][c]
    uint64_t *const bar = reinterpret_cast<uint64_t *>(T2 + 31 * 16);
    constexpr uint32_t AHEAD_BYTES = kAhead * 512 * sizeof(float2);
    auto ahead = [&](int64_t s) {
        mbar_expect_tx(bar, AHEAD_BYTES);
        tma_load_1d(P, a.in + s * kN, AHEAD_BYTES, bar);
    };
    grid_launch_dependents();
    if (tid < 31 * 16) T2[tid] = __ldg(a.tw + kTw2 + tid);  // (S2 reads it after S1's barrier)
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    grid_dependency_wait();
    if (tid == 0 && (int64_t)blockIdx.x < a.nseg) ahead(blockIdx.x);
    uint32_t par = 0;
    __syncthreads();
    const int a2 = tid >> 4, c2 = tid & 15, o2 = 512 * a2 + (c2 ^ (a2 & 15));
    const int a3 = tid & 31, x3 = a3 & 15, o3 = 512 * a3;
    for (int64_t s = blockIdx.x; s < a.nseg; s += gridDim.x) {
        float2 v[32];
        {  // S1
            const float2 *const x = a.in + s * kN + tid;
#pragma unroll
            for (int r = kAhead; r < 32; ++r) v[r] = x[512 * r];
            mbar_wait(bar, par, a.err);
            par ^= 1;
#pragma unroll
            for (int r = 0; r < kAhead; ++r) v[r] = P[512 * r + tid];
            float2 wb[8], wa[4];  // w_n^{j b}, w_n^{8 j a}
#pragma unroll
            for (int i = 1; i < 8; ++i) wb[i] = __ldg(a.tw + (i - 1) * 512 + tid);
#pragma unroll
            for (int i = 1; i < 4; ++i) wa[i] = __ldg(a.tw + (i + 6) * 512 + tid);
            dft<32, S>(v);
#pragma unroll
            for (int r = 0; r < 32; ++r) {
                if (r) v[r] = twmul<S>(v[r], r < 8 ? wb[r] : (r & 7) ? cmul(wa[r >> 3], wb[r & 7]) : wa[r >> 3]);
                sm[512 * r + (tid ^ (r & 15))] = v[r];
            }
        }
        __syncthreads();
        if (tid == 0 && s + gridDim.x < a.nseg) {  // the next segment: the rows ahead, the others to L2
            fence_proxy_async();
            ahead(s + gridDim.x);
            prefetch_l2_bulk(a.in + (s + gridDim.x) * kN + kAhead * 512, (32 - kAhead) * 512 * (uint32_t)sizeof(float2));
        }
        {  // S2
#pragma unroll
            for (int r = 0; r < 32; ++r) v[r] = sm[o2 + 16 * r];
            dft<32, S>(v);
#pragma unroll
            for (int q = 0; q < 32; q += 8) {  // (twiddles in batches: a shared load stays behind a shared store)
                float2 w[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (q + i) w[i] = T2[(q + i - 1) * 16 + c2];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (q + i) v[q + i] = twmul<S>(v[q + i], w[i]);
                    sm[o2 + 16 * (q + i)] = v[q + i];
                }
            }
        }
        __syncthreads();
        {  // S3: butterflies (k_a, k_b = tid / 32 + 16 q)
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int c = 0; c < 16; ++c) v[16 * q + c] = sm[o3 + 16 * ((tid >> 5) + 16 * q) + (c ^ x3)];
            __syncthreads();  // every point read: the next segment may land
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                dft<16, S>(v + 16 * q);
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const float2 y = cscale(v[16 * q + c], a.scale);
                    const int64_t o = s * kN + tid + 512 * q + 1024 * c;
                    if (a.out_power) static_cast<float *>(a.out)[o] = power_of(y);
                    else static_cast<float2 *>(a.out)[o] = y;
                }
            }
        }
    }
}

template <int S>
cudaError_t one_sm_t(const OneSmArgs &a, cudaStream_t st)
{
    auto k = k_one_sm<S>;
    static bool configured_dev[kMaxDevices] = {};  // per instantiation and device
    bool &configured = configured_dev[current_device_slot()];
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    // A few segments: launched with programmatic stream serialization, so that the
    // launch and the tables overlap the previous kernel (calls of 1 to 75 segments,
    // one after the other: 10.4 -> 8.0 us; the 4-CTA cluster kernel 9.0 up to 24).
    // More segments take the SMs in an ordinary launch: a CTA that waits holds an
    // SM that another stream's kernels could use.
    const int64_t sms = device_sm_count();
    if (a.nseg <= sms / 2) return launch_programmatic(k, (unsigned)a.nseg, kT, kSmem, st, a);
    k<<<(unsigned)(a.nseg < sms ? a.nseg : sms), kT, kSmem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

// w_n^{j b} (b = 1..7), w_n^{8 j a} (a = 1..3) over j < 512; w_512^{c r} [r-1][16]
void one_sm_tables(std::vector<float2> &h)
{
    h.resize(kTw);
    for (int i = 1; i < 8; ++i) host_roots(h.data() + (i - 1) * 512, 512, kN, i);
    for (int i = 1; i < 4; ++i) host_roots(h.data() + (i + 6) * 512, 512, kN, 8 * i);
    for (int r = 1; r < 32; ++r) host_roots(h.data() + kTw2 + (r - 1) * 16, 16, 512, r);
}

cudaError_t launch_one_sm(int sign, const OneSmArgs &a, cudaStream_t st)
{
    if (a.nseg <= 0) return cudaSuccess;
    return sign < 0 ? one_sm_t<-1>(a, st) : one_sm_t<1>(a, st);
}

}  // namespace fftseg
