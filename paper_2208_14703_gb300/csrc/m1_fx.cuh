// FP64 work on the integer pipe: the M1 closure and the neighbour sums of a cell
// in 64-bit fixed point.
//
// GB300 issues one FP64 warp instruction per 64 clocks and SM partition, a
// 32 x 32 + 64-bit multiply-add per 2.6 and a 64-bit add per 4 (measured).  The
// stencil kernels were bound by the FP64 pipe with nearly 90% of their issue
// slots idle.  A cell's closure and its contribution to its neighbours need no
// exponents of their own: with |F| <= c E every quantity (F / c, the tensor
// P) is at most E in size, so the six numbers of a cell fit one block: an
// exponent, E's, and 64-bit significands relative to it.  Products keep 62 bits,
// sums are exact, so the results carry 57 bits or more relative to E where FP64
// carried 53 with a rounding per operation: no precision is lost.
//
// Blocks are formed for regular cells only (fx_regular below: E a normal number
// of ordinary size, |F| <= c E up to a slack); a warp that meets another cell
// takes the FP64 form of its strip instead, which is the one that handles
// infinities, NaN and inadmissible states.
//
// The functions are host code too, so that their arithmetic can be checked
// without a GPU (the host takes IEEE results where the device takes the
// hardware's approximate reciprocals; both are seeds of the same iterations).
#pragma once
#include <cmath>
#include <cuda_runtime.h>

#include "m1_device.cuh"

namespace m1 {

typedef long long i64;
typedef unsigned long long u64;

__host__ __device__ __forceinline__ u64 bits_of_double(double x)
{
#ifdef __CUDA_ARCH__
    return (u64)__double_as_longlong(x);
#else
    u64 b;
    memcpy(&b, &x, sizeof b);
    return b;
#endif
}

__host__ __device__ __forceinline__ double double_of_bits(u64 b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((i64)b);
#else
    double x;
    memcpy(&x, &b, sizeof x);
    return x;
#endif
}

// seeds: about 2^-22 relative
__host__ __device__ __forceinline__ float seed_rcp(float x)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / x;
#endif
}

__host__ __device__ __forceinline__ float seed_rsqrt(float x)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / sqrtf(x);
#endif
}

__host__ __device__ __forceinline__ float seed_sqrt(float x)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return sqrtf(x);
#endif
}

// a * b + c of 32-bit a, b and 64-bit c (one instruction)
__host__ __device__ __forceinline__ i64 madw(int a, int b, i64 c) { return (i64)a * b + c; }

// A number |x| < 2^62 split at bit 31 (h signed, 0 <= l < 2^31), so that the
// partial products are signed 32 x 32 bits.
struct Split {
    int h, l;
};
__host__ __device__ __forceinline__ Split split62(i64 x)
{
    return Split{ (int)(x >> 31), (int)((unsigned)x & 0x7fffffffu) };
}

// a b / 2^62 (+ c), |a|, |b| < 2^62, within 2 units
__host__ __device__ __forceinline__ i64 mul62(Split a, Split b, i64 c = 0)
{
    const i64 mid = madw(a.h, b.l, madw(a.l, b.h, 0));
    return madw(a.h, b.h, mid >> 31) + c;
}

__host__ __device__ __forceinline__ i64 sqr62(Split a)
{
    const i64 mid = madw(a.h, a.l, 0);
    return madw(a.h, a.h, mid >> 30);
}

// a b / 2^62 to the nearest, ties to even, |a| < 2^61, 0 <= b < 2^62: odd in a and exact at
// zero, so that a scaled pair of neighbours (unequal cell sides) keeps the signs and the zeros
// of the sums it scales and adds no bias to a total.
__host__ __device__ __forceinline__ i64 fx_product(i64 a, Split b)
{
    const i64 s = a >> 63;
    const Split m = split62((a ^ s) - s);
    const i64 mid = madw(m.h, b.l, madw(m.l, b.h, madw(m.l, b.l, 0) >> 31));
    i64 v = madw(m.h, b.h, mid >> 31);
    v += (((unsigned)mid & 0x7fffffffu) + 0x3fffffffu + ((unsigned)v & 1u)) >> 31;
    return (v ^ s) - s;
}

// a cell's block: values v = m 2^(e - 60), F over c
struct FxCell {
    int e;
    i64 E, Fx, Fy, Pxx, Pxy, Pyy;
};

// exponents (biased) of the E a block can hold: 2^-500 .. 2^500
constexpr unsigned kFxMinExp = 1023 - 500, kFxMaxExp = 1023 + 500;

// The significand of x relative to 2^(be - 1023) at scale 2^61, truncated; the
// biased exponent of x is at most be (d >= 0), subnormals and zero give 0.
__host__ __device__ __forceinline__ i64 fx_align(u64 bits, int d)
{
    const u64 m = ((bits & 0xfffffffffffffull) | 0x10000000000000ull) << 9;
    const i64 v = (i64)(d > 63 ? 0 : m >> d);
    const i64 s = (i64)bits >> 63;
    return (v ^ s) - s;
}

// sigma = sqrt(xi) (scale 2^60; xi at 2^60, in [x^2/4, x^2]) and, returned, 3/2 D =
// 3/2 / (x + sigma) at scale 2^62, x at 2^61.
__host__ __device__ __forceinline__ i64 fx_sigma_d(i64 xE, i64 xi, i64& sg)
{
    // sigma = sqrt(xi): a 30-bit start s0 from the seed y of 1/sqrt(xi), then two
    // Newton corrections sigma += (xi - sigma^2) y / 2, exact residuals
    const float xif = (float)(int)(xi >> 32) * 0x1p-28f;
    const float yf = seed_rsqrt(xif);
    const int Y = (int)(yf * 0x1p29f);                         // y <= 2
    const float sf = xif * yf;
    const int s0 = (int)(sf * 0x1.fffffcp29f);                  // < 2^31 (sigma < 2 up to rounding)
    const i64 t0 = xi - madw(s0, s0, 0);                       // scale 2^60, |t0| < 2^42
    const i64 d0 = madw((int)(t0 >> 12), Y, 0) >> 18;          // t0 y / 2, scale 2^60
    sg = ((i64)s0 << 30) + d0;
    const i64 t1 = xi - sqr62(split62(sg << 1));
    sg += madw((int)t1, Y, 0) >> 30;
    const i64 hx = xE >> 2;                                    // x / 2 at scale 2^60
    sg = sg > hx ? sg : hx;
    // D = 1 / (x + sigma), scale 2^62, from the seed r: D = r (1 + d + d^2),
    // d = 1 - (x + sigma) r, less 2^-57 so that 3/2 D stays below 2^62
    const i64 w = (xE >> 1) + sg;                              // scale 2^60, in [1.5, 4)
    const float rf = seed_rcp((float)(int)(w >> 32) * 0x1p-28f);
    const int Rr = (int)(rf * 0x1p31f);                        // r <= 2/3
    const Split sw = split62(w);
    const i64 d = ((1ll << 60) - 8) - madw(sw.h, Rr, madw(sw.l, Rr, 0) >> 31);
    const Split sd = split62(d);                               // |d| < 2^39
    const i64 rd = madw(sd.h, Rr, madw(sd.l, Rr, 0) >> 31);    // r d, scale 2^60
    const i64 rdd = madw((int)(d >> 22), (int)(rd >> 22), 0) >> 16;
    const i64 D = ((i64)Rr << 31) + ((rd + rdd) << 2);
    return D + (D >> 1);
}

// The closure of Eq. (5) and the cell's block, from E and F / c.  With x = E and
// sigma = sqrt(x^2 - 3/4 |F/c|^2) >= x/2 it reads
//   P = (2 sigma - x)/3 I + 3/2 (F/c)(F/c)^T / (x + sigma),
// the form of closure() multiplied through by E: one square root and one
// reciprocal, no division by E, smooth at F = 0.  Returns false when the cell is
// not regular (the block is then meaningless).
__host__ __device__ __forceinline__ bool fx_stage(double E, double Fx, double Fy, FxCell& o)
{
    const u64 be = bits_of_double(E), bx = bits_of_double(Fx), by = bits_of_double(Fy);
    const unsigned te = (unsigned)(be >> 52);                  // sign included
    const int dx = (int)te - (int)((unsigned)(bx >> 52) & 0x7ffu);
    const int dy = (int)te - (int)((unsigned)(by >> 52) & 0x7ffu);
    bool ok = te - kFxMinExp <= kFxMaxExp - kFxMinExp && dx >= 0 && dy >= 0;
    // scale 2^61: x in [1, 2), |F / c| < 2
    const i64 xE = (i64)(((be & 0xfffffffffffffull) | 0x10000000000000ull) << 9);
    const i64 xF = fx_align(bx, dx), yF = fx_align(by, dy);
    const Split sE = split62(xE), sX = split62(xF), sY = split62(yF);
    // scale 2^60: x^2 and |F/c|^2
    const i64 E2 = sqr62(sE);
    const i64 midF = madw(sX.h, sX.l, madw(sY.h, sY.l, 0));
    const i64 F2 = madw(sX.h, sX.h, madw(sY.h, sY.h, midF >> 30));
    ok = ok && F2 <= E2 + (E2 >> 10);
    // xi = x^2 - 3/4 |F/c|^2 in [x^2/4, x^2], scale 2^60
    i64 xi = E2 - F2 + (F2 >> 2);
    const i64 q2 = E2 >> 2;
    xi = xi > q2 ? xi : q2;
    i64 sg;
    const Split sD = split62(fx_sigma_d(xE, xi, sg));          // 3/2 D, scale 2^62
    // (2 sigma - x) / 3, scale 2^60: the factor is 2^61 / 3
    constexpr i64 third = 768614336404564651ll;
    const i64 iso = mul62(split62((sg << 2) - xE), split62(third));
    // 3/2 D F/c at scale 2^61, the tensor at scale 2^60
    const Split gx = split62(mul62(sX, sD)), gy = split62(mul62(sY, sD));
    o.Pxx = mul62(gx, sX, iso);
    o.Pxy = mul62(gx, sY);
    o.Pyy = mul62(gy, sY, iso);
    o.E = xE >> 1;
    o.Fx = xF >> 1;
    o.Fy = yF >> 1;
    o.e = (int)te - 1023;
    return ok;
}

// The double nearest s 2^(e - 58), ties to even; e within the blocks' exponents, |s| < 2^63.
// (Sums of blocks whose low bits are mostly zero tie often: rounding those up gave the
// total energy a drift of 2^-58 a sweep.)
__host__ __device__ __forceinline__ double fx_double(i64 s, int e)
{
    const u64 sign = (u64)s & 0x8000000000000000ull;
    u64 m = (u64)(s < 0 ? -s : s);
    if (m == 0) return 0.0;
#ifdef __CUDA_ARCH__
    const int z = __clzll((i64)m);
#else
    const int z = __builtin_clzll(m);
#endif
    m <<= z;                                                   // bit 63 set: value m 2^(e - 58 - z)
    const u64 q = m >> 11;                                     // 53 bits (2^53 carries into the exponent)
    m = q + ((((unsigned)m & 0x7ffu) + ((unsigned)q & 1u) + 0x3ffu) >> 11);
    return double_of_bits(sign | (m + ((u64)(1023 + 63 - 58 - 1 - z + e) << 52)));
}

// Arithmetic right shift by n >= 0 (63 and more: the sign).
__host__ __device__ __forceinline__ i64 fx_sar(i64 x, int n) { return x >> (n < 63 ? n : 63); }

// x rounded toward zero to FP32: values below its normal range give 0, above it
// (and NaN) infinity.  For seeds, corrections and decisions with a margin.
__host__ __device__ __forceinline__ float narrow_rz(double x)
{
    const u64 b = bits_of_double(x);
    const unsigned mag = (unsigned)(b >> 32) & 0x7fffffffu;
    unsigned f = (unsigned)((b & 0x7fffffffffffffffull) >> 29) - (896u << 23);
    f = mag < (897u << 20) ? 0u : (mag >= (1151u << 20) ? 0x7f800000u : f);
    return float_of_bits(f | ((unsigned)(b >> 32) & 0x80000000u));
}

// The significand of a positive normal x at scale 2^61, and its exponent.
__host__ __device__ __forceinline__ i64 fx_significand(double x, int& e)
{
    const u64 b = bits_of_double(x);
    e = (int)(b >> 52) - 1023;
    return (i64)(((b & 0xfffffffffffffull) | 0x10000000000000ull) << 9);
}

// The root T of C T + K T^4 = R (C, K, R > 0) and T^4: Newton in FP32 to about
// 2e-7 (from `seed` when that is positive and a quarter
// or less off), then two
// corrections whose residuals are formed in fixed point relative
// to R (both terms are positive and sum to R) and whose quotients are FP32 (each
// needs only the digits it adds).  With t = T 2^(61 - eT) the powers are
// t^2 = T2 2^62, T2^2 = T4 2^62.  The residual is good to 2^-55 R, hence T to
// about 2^-55 and T^4 to 2^-53.  False where FP32 cannot hold or seed the problem.
__host__ __device__ __forceinline__ bool fx_quartic(double C, double K, double R, double& Tout,
                                                    double& T4out, float seed = 0.0f)
{
    const float Cf = narrow_rz(C), Kf = narrow_rz(K), Rf = narrow_rz(R);
    const float K4 = 4.0f * Kf;
    // one Newton step; the root then lies within 1.5 dT^2 / T (g'' T <= 3 g')
    auto newton = [&](float T, float& dT) {
        const float T3 = T * T * T;
        const float g = fmaf(Kf, T3 * T, Cf * T) - Rf;
        dT = g * seed_rcp(fmaf(K4, T3, Cf));
        return T - dT;
    };
    float dT = 0.0f, T = seed > 0.0f ? newton(seed, dT) : 0.0f;
    bool ok = seed > 0.0f && fabsf(dT) <= 3e-4f * T;
    if (!(seed > 0.0f && fabsf(dT) <= 0.25f * seed))
        T = fminf(Rf * seed_rcp(Cf), seed_sqrt(seed_sqrt(Rf * seed_rcp(Kf))));
    for (int it = 0; it < 40 && !ok; ++it) {
        T = newton(T, dT);
        ok = fabsf(dT) <= 3e-4f * T;
    }
    const unsigned bt = bits_of_float(T);
    // A significand at its upper end (T just below a power of two, such as a gas at rest
    // near T = 1) is taken as one below 1 at the next exponent, so that the corrections
    // (below 2^-18 T) keep it under 2^62.
    const int up = (bt & 0x7fffffu) >= 0x7fff00u ? 1 : 0;
    const int eT = (int)(bt >> 23) - 127 + up;                 // sign set: out of range below
    int eC, eK, eR;
    const i64 mC = fx_significand(C, eC), mR = fx_significand(R, eR);
    const Split sC = split62(mC), sK = split62(fx_significand(K, eK));
    const float dg = fmaf(K4, T * T * T, Cf);
    // 2^(eR - eT) / g' <= 4
    ok = ok && eT > -60 && eT < 60 && eR > -120 && eR < 120 && eR - eT > -120 && eR - eT < 120 &&
         dg > 1e-35f && dg < 1e35f;
    const float q = float_of_bits((unsigned)((ok ? eR - eT : 0) + 127) << 23) * seed_rcp(dg);
    const int nC = eR - eC - eT + 4, nK = eR - eK - 4 * eT + 1;
    ok = ok && nC >= 0 && nK >= 0;
    i64 m = (i64)((bt & 0x7fffffu) | 0x800000u) << (38 - up), T4 = 0;
    float d = 0.0f;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int pass = 0; pass < 2; ++pass) {
        const Split sm = split62(m);
        T4 = sqr62(split62(sqr62(sm)));
        const i64 g = fx_sar(mul62(sC, sm), nC) + fx_sar(mul62(sK, split62(T4)), nK) - (mR >> 5);
        if (pass == 0) {                                       // |g| < 2^38, in units 2^(eR - 56)
            const i64 gs = g >> 8;
            ok = ok && gs < 0x7fffffffll && gs > -0x7fffffffll;
            d = (float)(int)gs * q * 2.0f;                     // in units 2^12 of m
            ok = ok && fabsf(d) < 0x1p30f;
            m -= (i64)(int)(ok ? d : 0.0f) << 12;
        } else {
            ok = ok && g < 0x7fffffffll && g > -0x7fffffffll;
            d = (float)(int)g * q * 32.0f;
            ok = ok && fabsf(d) < 0x1p30f;
            d = ok ? d : 0.0f;
        }
    }
    // T^4 at the corrected root: T4 (1 - 4 d / m), with 4 T4 / m = t^3 / 2, t = T / 2^eT
    const float t = float_of_bits((bt & 0x7fffffu) | (0x3f800000u - ((unsigned)up << 23)));
    T4 -= (i64)(int)(d * t * t * t * 0.5f);
    m -= (i64)(int)d;
    T4out = fx_double(T4, ok ? 4 * eT : 0);
    // m in [2^60, 2^62) at exponent eT
    const int z = m < (1ll << 61) ? 1 : 0;
    const u64 r = ((u64)(m << z) >> 9) + (((u64)(m << z) >> 8) & 1);
    Tout = double_of_bits(r + ((u64)(1022 + (ok ? eT : 0) - z) << 52));
    return ok;
}

// What a cell adds to its neighbour's sums across one face (Eq. (9) with F over
// c and a common factor c dt / (2 h) taken out): E +- F_d, F_x +- P_xd, F_y +- P_yd.
struct FxFlux {
    int e;
    i64 E, Fx, Fy;
};

}  // namespace m1
