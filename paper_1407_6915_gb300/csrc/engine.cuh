// Register/shared-memory FFT engine shared by the sm_103a kernels.
//
// A "tile" is W lines of L points each (L, W powers of two).  Each of the T
// threads of a CTA holds V = W*L/T points in registers.  A length-L DFT runs
// as Stockham autosort stages of radix 16 (then one radix 2/4/8 stage for the
// remainder).  Stage with radix R after Ns points have been combined:
//   butterfly (c, j), j < L/R, reads  a_r = line_c[j + r*L/R],
//   multiplies a_r by w_{Ns*R}^{(j mod Ns)*r}, takes the R-point DFT, and
//   writes  line_c[(j/Ns)*Ns*R + (j mod Ns) + r*Ns] = A_r.
// The first stage reads global memory and the last writes it, both in the
// coalesced "j + r*L/R" order; stages in between exchange through shared
// memory.  This is the Cooley-Tukey FFT (Sec. I of the paper) in the
// self-sorting Stockham arrangement, so the output is in natural order.
//
// w_M^m = exp(sigma * 2 pi i m / M); tables hold the forward value
// (cos, -sin), evaluated in double on the host and rounded once to float.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#define FDEV __device__ __forceinline__
#define HDEV __host__ __device__ __forceinline__

// Self-checking build (compiled with -DFFTSEG_DEBUG): FFTSEG_CHECK(cond, err)
// is cond, and when cond is false it also sets bit 8 of *err, which
// fftseg_plan_check reports.  The caller then keeps the access inside its
// buffer (it is skipped or redirected), so a bad index is recorded, never
// performed: nothing traps.  In the normal build it is `true` and costs
// nothing.
#ifdef FFTSEG_DEBUG
#define FFTSEG_CHECK(cond, err) ((cond) ? true : (atomicOr((err), 8), false))
#else
#define FFTSEG_CHECK(cond, err) true
#endif

namespace fftseg {

// Complex additions and real-scalar multiply-adds act on both components
// alike, so they take the packed FP32 instructions of sm_100+ (two operations
// per lane and issue slot, each rounded as its scalar form).  The butterflies
// below are arranged so that most of their work is of this kind: the lane-line
// kernel at n = 2^16 is short of issue slots and of warps to hide latency: its
// 4 GiB transform measured 2.09 ms with scalar butterflies, 1.91 ms with the
// additions packed and 1.90 ms with the rotations below folded into them.
#ifdef __CUDA_ARCH__
FDEV unsigned long long pack2(float2 a)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
FDEV float2 unpack2(unsigned long long r)
{
    float2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
    return a;
}
#endif

HDEV float2 cadd(float2 a, float2 b)
{
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
#else
    return make_float2(a.x + b.x, a.y + b.y);
#endif
}

HDEV float2 csub(float2 a, float2 b)
{
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
#else
    return make_float2(a.x - b.x, a.y - b.y);
#endif
}

// a * s, s real
HDEV float2 cscale(float2 a, float s)
{
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(make_float2(s, s))));
    return unpack2(r);
#else
    return make_float2(a.x * s, a.y * s);
#endif
}

// a.x * s.x, a.y * s.y
HDEV float2 cmul_each(float2 a, float2 s)
{
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(s)));
    return unpack2(r);
#else
    return make_float2(a.x * s.x, a.y * s.y);
#endif
}

// a * s + b, s real
HDEV float2 cfma(float2 a, float s, float2 b)
{
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(make_float2(s, s))), "l"(pack2(b)));
    return unpack2(r);
#else
    return make_float2(a.x * s + b.x, a.y * s + b.y);
#endif
}

// a * w for the forward table entry w; the inverse uses conj(w).
template <int S>
HDEV float2 twmul(float2 a, float2 w)
{
    if (S < 0) return make_float2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
    return make_float2(a.x * w.x + a.y * w.y, a.y * w.x - a.x * w.y);
}

HDEV float2 cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }

// a * (sigma i)
template <int S>
HDEV float2 mul_si(float2 a)
{
    return S < 0 ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
}

constexpr float kC8 = 0.70710678118654752440f;   // cos(pi/4)
constexpr float kC16a = 0.92387953251128675613f;  // cos(pi/8)
constexpr float kC16b = 0.38268343236508977173f;  // sin(pi/8)

// A rotation by theta is cos(theta) (a + i tan(theta) a) or sin(theta)
// (cot(theta) a + i a).  rot_u gives the factor in brackets, with the tangent
// (or cotangent) t of theta <= pi/4 (or >= pi/4), at most 1 in size: two
// multiply-adds instead of two multiplications and two multiply-adds, and the
// cosine (or sine) left over goes into the packed additions that follow as
// their multiplier (one rounding less as well).
//   COT = false: a + sigma i t a;   COT = true: t a + sigma i a
template <bool COT, int S>
HDEV float2 rot_u(float2 a, float t)
{
    const float st = (float)S * t;
    if (COT) {
        if (S < 0) return make_float2(t * a.x + a.y, t * a.y - a.x);
        return make_float2(t * a.x - a.y, t * a.y + a.x);
    }
    return make_float2(a.x - st * a.y, a.y + st * a.x);
}

constexpr float kT8 = 0.41421356237309504880f;  // tan(pi/8) = cot(3 pi/8)

template <int S>
HDEV void dft2(float2 &a, float2 &b)
{
    const float2 t = a;
    a = cadd(t, b);
    b = csub(t, b);
}

// X_k = sum_j v_j w_4^{jk}, in place, natural order.
template <int S>
HDEV void dft4(float2 &v0, float2 &v1, float2 &v2, float2 &v3)
{
    const float2 a0 = cadd(v0, v2), a1 = csub(v0, v2);
    const float2 a2 = cadd(v1, v3), a3 = mul_si<S>(csub(v1, v3));
    v0 = cadd(a0, a2);
    v2 = csub(a0, a2);
    // (scalar: the quarter turn swaps the components, which an unpacked
    // addition takes as it is)
    v1 = make_float2(a1.x + a3.x, a1.y + a3.y);
    v3 = make_float2(a1.x - a3.x, a1.y - a3.y);
}

// dft4 of (v0, v1, c v2, v3 and v1 scaled by d): v0 + c v2 etc., with the real
// factors c of v2 and d of (v1, v3) folded into the additions.
template <int S>
HDEV void dft4_scaled(float2 &v0, float2 &v1, float2 &v2, float2 &v3, float c, float d)
{
    const float2 a0 = cfma(v2, c, v0), a1 = cfma(v2, -c, v0);
    const float2 a2 = cadd(v1, v3), a3 = mul_si<S>(csub(v1, v3));
    v0 = cfma(a2, d, a0);
    v2 = cfma(a2, -d, a0);
    v1 = make_float2(a3.x * d + a1.x, a3.y * d + a1.y);
    v3 = make_float2(a1.x - a3.x * d, a1.y - a3.y * d);
}

// 8 = 2 x 4: X_k = E_k + w_8^k O_k, X_{k+4} = E_k - w_8^k O_k
// (w_8 = cos(pi/4) (1 + sigma i), w_8^3 = cos(pi/4) (-1 + sigma i)).
template <int S>
HDEV void dft8(float2 *v)
{
    float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<S>(e0, e1, e2, e3);
    dft4<S>(o0, o1, o2, o3);
    o1 = rot_u<false, S>(o1, 1.f);
    o2 = mul_si<S>(o2);
    o3 = rot_u<true, S>(o3, -1.f);
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cfma(o1, kC8, e1);
    v[5] = cfma(o1, -kC8, e1);
    v[2] = make_float2(e2.x + o2.x, e2.y + o2.y);
    v[6] = make_float2(e2.x - o2.x, e2.y - o2.y);
    v[3] = cfma(o3, kC8, e3);
    v[7] = cfma(o3, -kC8, e3);
}

// 16 = 4 x 4 with j = 4 j1 + j2 and k = k1 + 4 k2:
//   Y[j2][k1] = w_16^{j2 k1} sum_{j1} v[4 j1 + j2] w_4^{j1 k1};
//   X[k1 + 4 k2] = sum_{j2} Y[j2][k1] w_4^{j2 k2}.
// The twiddles w_16^{j2 k1} as rot_u and a real factor: w^1 = cos(pi/8) (1 + i t),
// w^2 = cos(pi/4) (1 + i), w^3 = cos(pi/8) (t + i), w^6 = cos(pi/4) (-1 + i),
// w^9 = -w^1, t = tan(pi/8), i with the sign sigma.
template <int S>
HDEV void dft16(float2 *v)
{
#pragma unroll
    for (int j2 = 0; j2 < 4; ++j2) dft4<S>(v[j2], v[4 + j2], v[8 + j2], v[12 + j2]);
    // v[j2 + 4 k1] = Y[j2][k1] before the twiddle
    dft4<S>(v[0], v[1], v[2], v[3]);
    v[5] = rot_u<false, S>(v[5], kT8);
    v[6] = rot_u<false, S>(v[6], 1.f);
    v[7] = rot_u<true, S>(v[7], kT8);
    dft4_scaled<S>(v[4], v[5], v[6], v[7], kC8, kC16a);
    v[9] = rot_u<false, S>(v[9], 1.f);
    v[11] = rot_u<true, S>(v[11], -1.f);
    {
        const float2 b = mul_si<S>(v[10]);
        const float2 a0 = make_float2(v[8].x + b.x, v[8].y + b.y), a1 = make_float2(v[8].x - b.x, v[8].y - b.y);
        const float2 a2 = cadd(v[9], v[11]), a3 = mul_si<S>(csub(v[9], v[11]));
        v[8] = cfma(a2, kC8, a0);
        v[10] = cfma(a2, -kC8, a0);
        v[9] = make_float2(a3.x * kC8 + a1.x, a3.y * kC8 + a1.y);
        v[11] = make_float2(a1.x - a3.x * kC8, a1.y - a3.y * kC8);
    }
    v[13] = rot_u<true, S>(v[13], kT8);
    v[14] = rot_u<true, S>(v[14], -1.f);
    v[15] = rot_u<false, S>(v[15], kT8);
    {
        // v[15]'s factor is -cos(pi/8): its sum and difference with v[13] swap
        const float2 a0 = cfma(v[14], kC8, v[12]), a1 = cfma(v[14], -kC8, v[12]);
        const float2 a2 = csub(v[13], v[15]), a3 = mul_si<S>(cadd(v[13], v[15]));
        v[12] = cfma(a2, kC16a, a0);
        v[14] = cfma(a2, -kC16a, a0);
        v[13] = make_float2(a3.x * kC16a + a1.x, a3.y * kC16a + a1.y);
        v[15] = make_float2(a1.x - a3.x * kC16a, a1.y - a3.y * kC16a);
    }
    // v[4 k1 + k2] = X[k1 + 4 k2]; restore natural order
    float2 t[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) t[k] = v[4 * (k & 3) + (k >> 2)];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = t[k];
}

// a * w_32^M, w_32 = exp(sigma 2 pi i / 32), M = 0..15, from cos(M pi/16)
// and sin(M pi/16) (first-octant values c1 = cos(pi/16), s1 = sin(pi/16),
// c3 = cos(3 pi/16), s3 = sin(3 pi/16), and those of rot16)
template <int M, int S>
HDEV float2 rot32(float2 a)
{
    static_assert(M >= 0 && M < 16, "rot32 exponent");
    if constexpr (M == 0) return a;
    else if constexpr (M == 8) return mul_si<S>(a);
    else {
        constexpr float c1 = 0.98078528040323044913f, s1 = 0.19509032201612826785f;
        constexpr float c3 = 0.83146961230254523708f, s3 = 0.55557023301960222474f;
        constexpr float CS[16][2] = {{1.f, 0.f},      {c1, s1},        {kC16a, kC16b},  {c3, s3},
                                     {kC8, kC8},      {s3, c3},        {kC16b, kC16a},  {s1, c1},
                                     {0.f, 1.f},      {-s1, c1},       {-kC16b, kC16a}, {-s3, c3},
                                     {-kC8, kC8},     {-c3, s3},       {-kC16a, kC16b}, {-c1, s1}};
        constexpr float C = CS[M][0], Sn = CS[M][1];
        constexpr float s = (float)S;
        return make_float2(a.x * C - s * a.y * Sn, a.y * C + s * a.x * Sn);
    }
}

// e +- w_32^M o for M = 1..15: w_32^M = C (1 + sigma i t) for M <= 4 (t =
// tan(M pi/16)) and M >= 12 (C = cos(M pi/16) < 0), S (t + sigma i) between
// (t = cot(M pi/16), S = sin(M pi/16)); C and S are at least cos(pi/4) in size.
// C is the float above cos, not the nearest: the nearest floats of all three
// cosines and of cos(pi/4) lie below (by 1.7e-8 to 3.1e-8), which shrinks every
// output in step, and this error does not average out over a spectrum.  cos
// from above makes up for the rest: an emulated 32 x 32 transform in 32 bits
// has 1.02e-7 of error instead of 1.13e-7, its squared magnitudes on tones
// 6.5e-8 instead of 1.2e-7.
template <int M, int S>
HDEV void butterfly32(float2 e, float2 o, float2 &p, float2 &q)
{
    static_assert(M >= 1 && M < 16, "butterfly32 exponent");
    if constexpr (M == 8) {
        const float2 b = mul_si<S>(o);
        p = make_float2(e.x + b.x, e.y + b.y);
        q = make_float2(e.x - b.x, e.y - b.y);
    } else {
        // cos(pi/16), cos(pi/8), cos(3 pi/16), rounded up: see above
        constexpr float c1 = 0.98078531f, c2 = 0.92387956f, c3 = 0.83146966f;
        constexpr float t1 = 0.19891236737965800691f, t3 = 0.66817863791929891999f;   // tan(pi/16), tan(3 pi/16)
        constexpr int Q = M < 8 ? M : 16 - M, O = Q <= 4 ? Q : 8 - Q;  // O: distance to the nearest axis
        constexpr float T = O == 1 ? t1 : O == 2 ? kT8 : O == 3 ? t3 : 1.f;
        constexpr float C = O == 1 ? c1 : O == 2 ? c2 : O == 3 ? c3 : kC8;
        constexpr bool COT = Q > 4;
        // M > 8: cos < 0 < sin: -C (1 - sigma i T) or S (-T + sigma i)
        const float2 u = rot_u<COT, S>(o, M < 8 ? T : -T);
        constexpr float F = (!COT && M > 8) ? -C : C;
        p = cfma(u, F, e);
        q = cfma(u, -F, e);
    }
}

// 32 = 2 x 16: X_k = E_k + w_32^k O_k, X_{k+16} = E_k - w_32^k O_k, with E, O
// the 16-point DFTs of the even and odd samples.
template <int S>
HDEV void dft32(float2 *v)
{
    float2 e[16], o[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        e[i] = v[2 * i];
        o[i] = v[2 * i + 1];
    }
    dft16<S>(e);
    dft16<S>(o);
    v[0] = cadd(e[0], o[0]);
    v[16] = csub(e[0], o[0]);
    butterfly32<1, S>(e[1], o[1], v[1], v[17]);
    butterfly32<2, S>(e[2], o[2], v[2], v[18]);
    butterfly32<3, S>(e[3], o[3], v[3], v[19]);
    butterfly32<4, S>(e[4], o[4], v[4], v[20]);
    butterfly32<5, S>(e[5], o[5], v[5], v[21]);
    butterfly32<6, S>(e[6], o[6], v[6], v[22]);
    butterfly32<7, S>(e[7], o[7], v[7], v[23]);
    butterfly32<8, S>(e[8], o[8], v[8], v[24]);
    butterfly32<9, S>(e[9], o[9], v[9], v[25]);
    butterfly32<10, S>(e[10], o[10], v[10], v[26]);
    butterfly32<11, S>(e[11], o[11], v[11], v[27]);
    butterfly32<12, S>(e[12], o[12], v[12], v[28]);
    butterfly32<13, S>(e[13], o[13], v[13], v[29]);
    butterfly32<14, S>(e[14], o[14], v[14], v[30]);
    butterfly32<15, S>(e[15], o[15], v[15], v[31]);
}

// Odd prime radix R = 3, 5, 7 by the pair sums and differences of the
// inputs: with A_k = v_k + v_{R-k}, B_k = v_k - v_{R-k} (k = 1..(R-1)/2),
//   X_0 = v_0 + sum_k A_k,
//   X_m, X_{R-m} = v_0 + sum_k cos(2 pi m k / R) A_k  +/-  sigma i sum_k sin(2 pi m k / R) B_k.
// odd_cos / odd_sin give cos and sin(2 pi q / R) for q = m k mod R (cos is
// even and sin odd in q, so q in 1..R-1 is enough).
template <int R>
HDEV constexpr float odd_cos(int q)
{
    // R = 3: cos(2 pi / 3); R = 5: cos(2 pi / 5), cos(4 pi / 5); R = 7: cos(2 pi k / 7), k = 1, 2, 3
    const int r = q <= R / 2 ? q : R - q;
    return R == 3 ? -0.5f
           : R == 5 ? (r == 1 ? 0.30901699437494742410f : -0.80901699437494742410f)
                    : (r == 1 ? 0.62348980185873353053f : r == 2 ? -0.22252093395631440429f : -0.90096886790241912624f);
}
template <int R>
HDEV constexpr float odd_sin(int q)
{
    const int r = q <= R / 2 ? q : R - q;
    const float v = R == 3 ? 0.86602540378443864676f
                    : R == 5 ? (r == 1 ? 0.95105651629515357212f : 0.58778525229247312917f)
                             : (r == 1 ? 0.78183148246802980871f : r == 2 ? 0.97492791218182360702f
                                                                          : 0.43388373911755812048f);
    return q <= R / 2 ? v : -v;
}

template <int R, int S>
HDEV void dft_odd(float2 *v)
{
    constexpr int H = (R - 1) / 2;
    float2 A[H], B[H];
    float2 x0 = v[0];
#pragma unroll
    for (int k = 0; k < H; ++k) {
        A[k] = cadd(v[k + 1], v[R - 1 - k]);
        B[k] = csub(v[k + 1], v[R - 1 - k]);
    }
    float2 X0 = x0;
#pragma unroll
    for (int k = 0; k < H; ++k) X0 = cadd(X0, A[k]);
    if constexpr (R == 3) {  // (the sine into the last additions: one rounding less)
        const float2 P = cfma(A[0], odd_cos<3>(1), x0), iB = mul_si<S>(B[0]);
        constexpr float sn = odd_sin<3>(1);
        v[1] = make_float2(iB.x * sn + P.x, iB.y * sn + P.y);
        v[2] = make_float2(P.x - iB.x * sn, P.y - iB.y * sn);
    } else {
#pragma unroll
        for (int m = 0; m < H; ++m) {
            float2 P = x0, Q = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < H; ++k) {
                const float c = odd_cos<R>(((m + 1) * (k + 1)) % R), sn = odd_sin<R>(((m + 1) * (k + 1)) % R);
                P = cfma(A[k], c, P);
                Q = cfma(B[k], sn, Q);
            }
            const float2 iQ = mul_si<S>(Q);  // sigma i Q
            v[m + 1] = make_float2(P.x + iQ.x, P.y + iQ.y);
            v[R - 1 - m] = make_float2(P.x - iQ.x, P.y - iQ.y);
        }
    }
    v[0] = X0;
}

// cos and sin(2 pi m / R) at compile time, by their Taylor series on
// [0, pi/4] (18 terms of the angle's powers; the argument's octant and the
// symmetries give the rest), rounded once to float.
__host__ __device__ constexpr double ct_series(double x, bool sine)
{
    double term = sine ? x : 1.0, sum = term;
    for (int i = sine ? 2 : 1; i < 18; i += 2) {
        term *= -x * x / ((double)i * (i + 1));
        sum += term;
    }
    return sum;
}
__host__ __device__ constexpr double ct_cos(int m, int R)
{
    m = ((m % R) + R) % R;
    if (2 * m > R) m = R - m;              // cos(2 pi - a) = cos(a)
    if (4 * m > R) return -ct_cos(R - 2 * m, 2 * R);  // cos(pi - a) = -cos(a)
    const double a = 6.283185307179586476925286766559 * m / R;
    if (8 * m <= R) return ct_series(a, false);
    return ct_series(1.5707963267948966192313216916398 - a, true);  // cos(a) = sin(pi/2 - a)
}
__host__ __device__ constexpr double ct_sin(int m, int R) { return ct_cos(4 * m - R, 4 * R); }  // sin(a) = cos(a - pi/2)

// a * w_R^M, w_R = exp(sigma 2 pi i / R)
template <int M, int R, int S>
HDEV float2 rot_const(float2 a)
{
    if constexpr (M % R == 0) return a;
    else if constexpr (4 * M == R) return mul_si<S>(a);
    else if constexpr (2 * M == R) return make_float2(-a.x, -a.y);
    else {
        constexpr float c = (float)ct_cos(M, R), s = (float)(S * ct_sin(M, R));
        return make_float2(a.x * c - a.y * s, a.y * c + a.x * s);
    }
}

// Composite radix R = A B with j = B j1 + j2, k = k1 + A k2, as dft16.
template <int A, int B, int S, int J2 = 1, int K1 = 1>
HDEV void dft_ab_twiddle(float2 *v)
{
    if constexpr (J2 < B) {
        v[K1 * B + J2] = rot_const<J2 * K1, A * B, S>(v[K1 * B + J2]);
        if constexpr (K1 + 1 < A) dft_ab_twiddle<A, B, S, J2, K1 + 1>(v);
        else dft_ab_twiddle<A, B, S, J2 + 1, 1>(v);
    }
}

template <int R, int S>
HDEV void dft(float2 *v);

template <int A, int B, int S>
HDEV void dft_ab(float2 *v)
{
#pragma unroll
    for (int j2 = 0; j2 < B; ++j2) {
        float2 t[A];
#pragma unroll
        for (int j1 = 0; j1 < A; ++j1) t[j1] = v[B * j1 + j2];
        dft<A, S>(t);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) v[B * k1 + j2] = t[k1];
    }
    dft_ab_twiddle<A, B, S>(v);
    float2 o[A * B];
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
        float2 t[B];
#pragma unroll
        for (int j2 = 0; j2 < B; ++j2) t[j2] = v[B * k1 + j2];
        dft<B, S>(t);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) o[k1 + A * k2] = t[k2];
    }
#pragma unroll
    for (int k = 0; k < A * B; ++k) v[k] = o[k];
}

// Composite radix R = A B with A, B coprime, without twiddles (the prime-factor
// algorithm of Good and Thomas): with j = B j1 + A j2 mod R, k = k1 mod A = k2
// mod B, w_R^{jk} = w_A^{j1 k1} w_B^{j2 k2}.
template <int A, int B, int S>
HDEV void dft_coprime(float2 *v)
{
    constexpr int R = A * B;
    float2 y[R], o[R];
#pragma unroll
    for (int j2 = 0; j2 < B; ++j2) {
        float2 t[A];
#pragma unroll
        for (int j1 = 0; j1 < A; ++j1) t[j1] = v[(B * j1 + A * j2) % R];
        dft<A, S>(t);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) y[k1 * B + j2] = t[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
        dft<B, S>(y + k1 * B);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) {
            // k = k1 mod A = k2 mod B (a compile-time search once unrolled)
            int k = k1;
#pragma unroll
            for (int i = 1; i < B; ++i)
                if ((k1 + A * i) % B == k2) k = k1 + A * i;
            o[k] = y[k1 * B + k2];
        }
    }
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = o[k];
}

template <int R, int S>
HDEV void dft(float2 *v)
{
    if constexpr (R == 2) dft2<S>(v[0], v[1]);
    else if constexpr (R == 6) dft_coprime<2, 3, S>(v);
    else if constexpr (R == 9) dft_ab<3, 3, S>(v);
    else if constexpr (R == 10) dft_coprime<2, 5, S>(v);
    else if constexpr (R == 12) dft_coprime<4, 3, S>(v);
    else if constexpr (R == 14) dft_coprime<2, 7, S>(v);
    else if constexpr (R == 15) dft_coprime<5, 3, S>(v);
    else if constexpr (R == 18) dft_coprime<2, 9, S>(v);
    else if constexpr (R == 24) dft_coprime<8, 3, S>(v);
    else if constexpr (R == 3 || R == 5 || R == 7) dft_odd<R, S>(v);
    else if constexpr (R == 4) dft4<S>(v[0], v[1], v[2], v[3]);
    else if constexpr (R == 8) dft8<S>(v);
    else if constexpr (R == 16) dft16<S>(v);
    else if constexpr (R == 32) dft32<S>(v);
}

// Radix schedule of a length-2^LOG_L line: radix 16 while possible, then one
// 2/4/8 stage.
template <int LOG_L, int STAGE>
struct StageInfo {
    static constexpr int NFULL = LOG_L / 4;
    static constexpr int REM = LOG_L % 4;
    static constexpr int NSTAGES = NFULL + (REM ? 1 : 0);
    static constexpr int LOG_R = (STAGE < NFULL) ? 4 : REM;
    static constexpr int R = 1 << LOG_R;
    static constexpr int LOG_NS = 4 * STAGE;
    static constexpr int NS = 1 << LOG_NS;
    static constexpr bool FIRST = STAGE == 0;
    static constexpr bool LAST = STAGE == NSTAGES - 1;
};

// Shared-memory slot of (line c, index i).  CFAST: lines interleaved
// (q = i*W + c); else line-major (q = c*L + i).  One pad slot every 2^PS
// slots keeps the strided accesses of the first stage conflict-free.
template <int LOG_L, int LOG_W, bool CFAST, int PS>
FDEV int smem_slot(int c, int i)
{
    const int q = CFAST ? ((i << LOG_W) + c) : ((c << LOG_L) + i);
    return q + (q >> PS);
}

template <int LOG_L, int LOG_W, int PS>
constexpr int smem_slots()
{
    return (1 << (LOG_L + LOG_W)) + ((1 << (LOG_L + LOG_W)) >> PS) + 1;
}

// Butterfly g of a stage with radix 2^LOG_R -> (line c, butterfly index j).
template <int LOG_L, int LOG_W, bool CFAST, int LOG_R>
FDEV void butterfly_coords(int g, int &c, int &j)
{
    if (CFAST) {
        c = g & ((1 << LOG_W) - 1);
        j = g >> LOG_W;
    } else {
        c = g >> (LOG_L - LOG_R);
        j = g & ((1 << (LOG_L - LOG_R)) - 1);
    }
}

// Stage twiddle tables.  Stage s > 0 (radix R, Ns = 16^s) multiplies element
// r of butterfly j by w_{Ns R}^{m r}, m = j mod Ns.  Its table holds these
// values r-major, [r-1][m], so that lanes with consecutive m read consecutive
// entries (or one broadcast entry); tables of stages 1, 2, ... follow each
// other.  stage_table_offset gives where stage s starts.
template <int LOG_L>
__host__ __device__ constexpr int stage_table_offset(int stage)
{
    int off = 0;
    for (int s = 1; s < stage; ++s) {
        const int lr = s < LOG_L / 4 ? 4 : LOG_L % 4;
        off += ((1 << lr) - 1) << (4 * s);
    }
    return off;
}

// Twiddle + DFT of one butterfly held in x[0..R).  tw: the stage tables of
// a length-L line (laid out as stage_table_offset gives).
template <int LOG_L, int STAGE, int S>
FDEV void apply_twiddles(float2 *x, int j, const float2 *__restrict__ tw)
{
    using I = StageInfo<LOG_L, STAGE>;
    if constexpr (!I::FIRST) {
        constexpr int OFF = stage_table_offset<LOG_L>(STAGE);
        const float2 *t = tw + OFF + (j & (I::NS - 1));
#pragma unroll
        for (int r = 1; r < I::R; ++r) x[r] = twmul<S>(x[r], __ldg(t + (r - 1) * I::NS));
    }
}

template <int LOG_L, int STAGE, int S>
FDEV void butterfly(float2 *x, int j, const float2 *__restrict__ tw)
{
    apply_twiddles<LOG_L, STAGE, S>(x, j, tw);
    dft<StageInfo<LOG_L, STAGE>::R, S>(x);
}

// Output index of element r of butterfly j.
template <int LOG_L, int STAGE>
FDEV int stockham_out_index(int j, int r)
{
    using I = StageInfo<LOG_L, STAGE>;
    return ((j >> I::LOG_NS) << (I::LOG_NS + I::LOG_R)) + (j & (I::NS - 1)) + (r << I::LOG_NS);
}

}  // namespace fftseg

// ------------------------------------------------------------------ TMA bulk
// 1-D bulk copies global -> shared (cp.async.bulk), completed on an mbarrier
// with transaction-byte accounting.  Every wait is bounded: after
// kSpinLimit polls the waiter records a timeout in *err and carries on, so a
// lost copy can never hang the GPU.
namespace fftseg {

constexpr uint32_t kSpinLimit = 1u << 24;

FDEV uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// 8-byte asynchronous copy global -> shared (cp.async; any 8-byte-aligned
// source).  src_bytes = 0 writes zeros and reads nothing.  Copies are grouped
// by cp_async_commit; cp_async_wait<N> returns once at most N of the calling
// thread's groups are pending, and the thread then sees its own copies
// (other threads' copies need a barrier after their waits).
FDEV void cp_async8(void *smem_dst, const void *gsrc, uint32_t src_bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_u32(smem_dst)), "l"(gsrc),
                 "r"(src_bytes)
                 : "memory");
}
FDEV void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
FDEV void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialization may start while the previous kernel in its stream is still
// running; grid_dependency_wait returns once that kernel has completed and
// its memory operations are visible (no global access of the data path may
// come before it), and launch_dependents lets the next such kernel start its
// own blocks as this one's leave.
FDEV void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
FDEV void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Bulk prefetch of global memory into L2 (16-byte aligned, bytes % 16 == 0).
// A hint only: lines fetched before a producer's writes to them are updated
// in L2 by those writes, so it may precede grid_dependency_wait.
FDEV void prefetch_l2_bulk(const void *src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

FDEV void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

FDEV void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// order this thread's earlier generic-proxy shared-memory accesses before
// later async-proxy (TMA) accesses
FDEV void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// order this thread's generic-proxy view of global memory (e.g. data another
// CTA published with a release) before its later async-proxy (TMA) reads
FDEV void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

// Tiled 3-D TMA store of one box from shared memory (16-byte aligned, dense
// box layout) to `tmap` at (x, y, z); tracked by bulk groups of this thread.
FDEV void tma_store_3d(const CUtensorMap *tmap, int x, int y, int z, const void *src)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                     reinterpret_cast<uint64_t>(tmap)),
                 "r"(x), "r"(y), "r"(z), "r"(smem_u32(src))
                 : "memory");
}

// tma_store_3d for a 4-D map, at (x, y, z, w)
FDEV void tma_store_4d(const CUtensorMap *tmap, int x, int y, int z, int w, const void *src)
{
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(
                     reinterpret_cast<uint64_t>(tmap)),
                 "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(src))
                 : "memory");
}

// tma_store_3d for a 5-D map, at (x, y, z, w, v)
FDEV void tma_store_5d(const CUtensorMap *tmap, int x, int y, int z, int w, int v, const void *src)
{
    asm volatile("cp.async.bulk.tensor.5d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4, %5}], [%6];" ::"l"(
                     reinterpret_cast<uint64_t>(tmap)),
                 "r"(x), "r"(y), "r"(z), "r"(w), "r"(v), "r"(smem_u32(src))
                 : "memory");
}

// wait until every committed bulk copy of this thread has completed its writes
FDEV void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// wait until every committed bulk store of this thread has read its source
FDEV void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// plain arrive (count 1) on an mbarrier
FDEV void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Release add at GPU scope: this thread's earlier memory operations, and those
// it has observed through synchronisation, are visible before the add.
FDEV void red_release_add(int *p, int v)
{
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Drop a 128-byte line from L2 without writing it back (its contents become
// undefined): for intermediate data that has been consumed.
FDEV void discard_l2_line(const void *p) { asm volatile("discard.global.L2 [%0], 128;" ::"l"(p) : "memory"); }

FDEV void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// dst (shared, 16-byte aligned) <- src (global, 16-byte aligned), bytes % 16 == 0
FDEV void tma_load_1d(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// Tiled 3-D TMA load of one box of `tmap` at element coordinates (x, y, z)
// into shared memory (16-byte aligned), completed on *bar.  x * 8 bytes must
// be a multiple of 16 (8-byte elements: x even).
FDEV void tma_load_3d(void *dst, const CUtensorMap *tmap, int x, int y, int z, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// Tiled 2-D TMA load of one box of `tmap` at (x, y) into shared memory with
// an L2 cache policy, completed on *bar (x * element size a multiple of 16).
FDEV void tma_load_2d_hint(void *dst, const CUtensorMap *tmap, int x, int y, uint64_t *bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}

// Tiled 4-D TMA load of one box of `tmap` at element coordinates (x, y, z, w)
// into shared memory, completed on *bar (x * element size a multiple of 16).
FDEV void tma_load_4d(void *dst, const CUtensorMap *tmap, int x, int y, int z, int w, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
        : "memory");
}

// L2 cache policy that leaves a line's eviction priority as it is (for data
// that is read twice, such as the overlap of consecutive frames).
FDEV uint64_t policy_evict_unchanged()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_unchanged.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// L2 cache policy: lines fetched or written under it are evicted first (for
// data streamed once, so that it does not displace data kept in L2).
FDEV uint64_t policy_evict_first()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// tma_load_3d with an L2 cache policy
FDEV void tma_load_3d_hint(void *dst, const CUtensorMap *tmap, int x, int y, int z, uint64_t *bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}

// tma_load_4d with an L2 cache policy
FDEV void tma_load_4d_hint(void *dst, const CUtensorMap *tmap, int x, int y, int z, int w, uint64_t *bar,
                           uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3, %4, %5}], [%6], %7;" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}

// tma_store_3d with an L2 cache policy
FDEV void tma_store_3d_hint(const CUtensorMap *tmap, int x, int y, int z, const void *src, uint64_t policy)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group.L2::cache_hint [%0, {%1, %2, %3}], [%4], %5;" ::"l"(
                     reinterpret_cast<uint64_t>(tmap)),
                 "r"(x), "r"(y), "r"(z), "r"(smem_u32(src)), "l"(policy)
                 : "memory");
}

// address of the same shared-memory variable in CTA `rank` of the cluster
FDEV uint32_t mapa_u32(uint32_t smem_addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
    return r;
}

FDEV void st_cluster_v2(uint32_t addr, float2 v)
{
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}

// Remote store into CTA-shared memory of a cluster peer that also credits 8
// bytes to the peer's mbarrier (st.async): the receiver learns of the data by
// waiting on its own barrier; no release fence is needed on the sender side.
FDEV void st_async_v2(uint32_t remote_addr, float2 v, uint32_t remote_bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(
                     remote_addr),
                 "f"(v.x), "f"(v.y), "r"(remote_bar)
                 : "memory");
}

// Bulk copy from this CTA's shared memory to a cluster peer's shared memory
// (both addresses 16-byte aligned, bytes % 16 == 0), completing on the peer's
// mbarrier.  dst and bar are shared::cluster addresses (mapa).
FDEV void dsmem_bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "r"(smem_u32(src)), "r"(bytes), "r"(bar)
                 : "memory");
}

FDEV void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }

// wait until every committed bulk copy of this thread has finished reading its source
FDEV void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// Cluster-wide execution barrier without memory ordering (arrive.relaxed):
// used where every thread has already consumed what it read.
FDEV void cluster_sync_relaxed()
{
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

// The two halves of cluster_sync_relaxed, for an arrive early and a wait late.
FDEV void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
FDEV void cluster_wait() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); }

FDEV bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Non-blocking test of phase `parity` of *bar.
FDEV bool mbar_test_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// GPU-scope acquire-release fence.
FDEV void fence_acq_rel_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// Wait for phase `parity` of *bar; false (and *err set) if it never completes.
FDEV bool mbar_wait(uint64_t *bar, uint32_t parity, int *err)
{
    for (uint32_t it = 0; it < kSpinLimit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    if (err) atomicOr(err, 1);
    return false;
}

}  // namespace fftseg
