// FP64 work on the integer pipe: the M1 closure and the neighbour sums of a cell
// in 64-bit fixed point.
//
// GB300 issues one FP64 warp instruction per 64 clocks and SM partition, a
// 32 x 32 + 64-bit multiply-add per 2.6 and a 64-bit add per 4 (measured).  The
// stencil kernels were bound by the FP64 pipe with nearly 90% of their issue
// slots idle.  A cell is held as a block: E, F_x / c and F_y / c as 64-bit significands,
// each with its own exponent, and the anisotropic part of the closure relative to them.
// With x = E, sigma = sqrt(x^2 - 3/4 |F/c|^2) and A = 3/2 (F/c)(F/c)^T / (x + sigma),
//   P = A + S I,  S = (x - tr A)/3 = (2 sigma - x)/3,
// so the flux of F_x across an x face is F_x +- A_xx +- S.  The sums of F and A are formed
// relative to the largest flux component of the stencil, the differences of S apart, in
// which like cells cancel exactly: a flux far below E (ahead of a front, across a grid
// uniform in that direction, transverse to a 1D grid) keeps its 53 bits, as it does in FP64.
// Products keep 62 bits, significands 58 (S: 61), sums are exact: each row of the sums carries
// its terms to 2^-56 or so where FP64 carried 2^-53 with a rounding per operation.
//
// Blocks are formed for regular cells only (fx_stage: E a normal number of ordinary size,
// |F| <= c E up to a slack, no flux component but zero below 2^-923); a warp that meets another
// cell takes the FP64 form of its strip instead, which is the one that handles
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

// v / 2^d rounded down, d a difference of exponents: any d >= 64, and any d < 0, which a
// regular cell excludes, leave the sign (the PTX shift's own rule).
__host__ __device__ __forceinline__ i64 fx_down(i64 v, int d)
{
#ifdef __CUDA_ARCH__
    i64 r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(d));
    return r;
#else
    return v >> ((unsigned)d < 63u ? d : 63);
#endif
}

// A cell's block, F over c.  Exponents are FP64's biased ones, e of E and ex, ey of the
// flux (in the halves of ef); the values are E = m 2^(e - 58), F_x = m 2^(ex - 58) and so
// on, less the bias, A_xx = m 2^(2 ex - e - 58), A_xy = m 2^(ex + ey - e - 58) and A_yy
// likewise; S = m 2^(e - 61).
struct FxCell {
    int e;
    unsigned ef;
    i64 E, Fx, Fy, Axx, Axy, Ayy, S;
};

// Exponents (biased) of the E a block can hold: 2^-500 .. 2^500; and the least of a flux
// component (2^-923, so that sums stay normal numbers), which zero is given too.
constexpr unsigned kFxMinExp = 1023 - 500, kFxMaxExp = 1023 + 500;
constexpr int kFxMinFlux = 100;

// A flux component's biased exponent and the size of its significand, scale 2^61; ok cleared
// where it is too small to hold.
__host__ __device__ __forceinline__ i64 fx_flux(u64 bits, int& t, bool& ok)
{
    t = (int)(bits >> 52) & 0x7ff;
    const i64 m = (i64)(((bits & 0xfffffffffffffull) | 0x10000000000000ull) << 9);
    if (t >= kFxMinFlux) return m;
    ok = ok && (bits << 1) == 0;
    t = kFxMinFlux;
    return 0;
}

// 3/2 D = 3/2 / (x + sigma) at scale 2^62, sigma = sqrt(xi), and S = (2 sigma - x)/3 at 2^61;
// x at scale 2^61, xi at 2^60 and in [x^2/4, x^2].
__host__ __device__ __forceinline__ i64 fx_d15(i64 xE, i64 xi, i64& S)
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
    i64 sg = ((i64)s0 << 30) + d0;
    const i64 t1 = xi - sqr62(split62(sg << 1));
    sg += madw((int)t1, Y, 0) >> 30;
    const i64 hx = xE >> 2;                                    // x / 2 at scale 2^60
    sg = sg > hx ? sg : hx;
    constexpr i64 third = 1537228672809129301ll;               // 2^62 / 3
    S = mul62(split62((sg << 2) - xE), split62(third));
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

// The closure of Eq. (5) and the cell's block, from E and F / c: one square root and one
// reciprocal, no division by E, smooth at F = 0, odd and even in the flux components as the
// closure is.  Returns false when the cell is not regular (the block is then meaningless).
__host__ __device__ __forceinline__ bool fx_stage(double E, double Fx, double Fy, FxCell& o)
{
    const u64 be = bits_of_double(E), bx = bits_of_double(Fx), by = bits_of_double(Fy);
    const unsigned te = (unsigned)(be >> 52);                  // sign included
    bool ok = te - kFxMinExp <= kFxMaxExp - kFxMinExp;
    int tx, ty;
    // scale 2^61: x in [1, 2), the sizes of the flux components too, each to its exponent
    const i64 xE = (i64)(((be & 0xfffffffffffffull) | 0x10000000000000ull) << 9);
    const i64 mX = fx_flux(bx, tx, ok), mY = fx_flux(by, ty, ok);
    const int dx = (int)te - tx, dy = (int)te - ty;
    ok = ok && dx >= 0 && dy >= 0;
    const Split sE = split62(xE), sX = split62(mX), sY = split62(mY);
    // scale 2^60: x^2 and |F/c|^2
    const i64 E2 = sqr62(sE);
    const i64 F2 = fx_down(sqr62(sX), 2 * dx) + fx_down(sqr62(sY), 2 * dy);
    ok = ok && F2 <= E2 + (E2 >> 10);
    // xi = x^2 - 3/4 |F/c|^2 in [x^2/4, x^2], scale 2^60
    i64 xi = E2 - F2 + (F2 >> 2);
    const i64 q2 = E2 >> 2;
    xi = xi > q2 ? xi : q2;
    const Split sD = split62(fx_d15(xE, xi, o.S));             // 3/2 D, scale 2^62
    // 3/2 D F/c at scale 2^61, A at scale 2^60, then 2^58 to the nearest
    const Split gx = split62(mul62(sX, sD)), gy = split62(mul62(sY, sD));
    const i64 nx = (i64)bx >> 63, ny = (i64)by >> 63, nxy = nx ^ ny;
    o.Axx = mul62(gx, sX, 2) >> 2;
    o.Axy = ((mul62(gx, sY, 2) >> 2) ^ nxy) - nxy;
    o.Ayy = mul62(gy, sY, 2) >> 2;
    o.E = xE >> 3;
    o.Fx = ((mX >> 3) ^ nx) - nx;
    o.Fy = ((mY >> 3) ^ ny) - ny;
    o.e = (int)te;
    o.ef = (unsigned)tx | (unsigned)ty << 16;
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

// What a cell adds to its neighbour's sums across one face (Eq. (9) with F over c and a
// common factor c dt / (2 h) taken out): E +- F_d, F_x +- A_xd and F_y +- A_yd, each at its own
// exponent, and S.  A cell gives to the east and north what it has there; what it gives to the
// west and south is held with the sign changed (-E + F_d, ...), so that rounding down, where a
// sum brings it to a larger exponent, rounds it up: the two faces of an axis together carry no
// bias, which a total over many sweeps would gather.  (A mirror image of a state exchanges the
// faces, so its sums may differ from the state's by that rounding.)
struct FxFlux {
    int e;
    unsigned ef;
    i64 E, I, X, Y;
};

// A cell's part of its x or y faces: F_d at E's exponent, A_xd and A_yd at those of the flux.
struct FxSide {
    i64 g, X, Y;
};
__host__ __device__ __forceinline__ FxSide fx_side_x(const FxCell& c)
{
    const int d = c.e - (int)(c.ef & 0xffffu);
    return FxSide{ fx_down(c.Fx, d), fx_down(c.Axx, d), fx_down(c.Axy, d) };
}
__host__ __device__ __forceinline__ FxSide fx_side_y(const FxCell& c)
{
    const int d = c.e - (int)(c.ef >> 16);
    return FxSide{ fx_down(c.Fy, d), fx_down(c.Axy, d), fx_down(c.Ayy, d) };
}

// Across the east or north faces, and (HIGH) the west or south ones.
template <bool HIGH>
__host__ __device__ __forceinline__ FxFlux fx_flux_of(const FxCell& c, const FxSide& s)
{
    return HIGH ? FxFlux{ c.e, c.ef, s.g - c.E, c.S, s.X - c.Fx, s.Y - c.Fy }
                : FxFlux{ c.e, c.ef, s.g + c.E, c.S, s.X + c.Fx, s.Y + c.Fy };
}

// The larger of each half of two pairs of flux exponents.
__host__ __device__ __forceinline__ unsigned fx_max2(unsigned a, unsigned b)
{
#ifdef __CUDA_ARCH__
    return __vmaxu2(a, b);
#else
    const unsigned lo = (a & 0xffffu) > (b & 0xffffu) ? a & 0xffffu : b & 0xffffu;
    return ((a >> 16) > (b >> 16) ? a >> 16 : b >> 16) << 16 | lo;
#endif
}

// A cell's neighbour sums: E, X and Y as in FxFlux at their exponents, and the differences
// of S that X and Y get, at the larger exponent of their pair (ex, ey).
struct FxSum {
    int e, ex, ey;
    unsigned ef;
    i64 E, X, Y, Ix, Iy;
};

// The two faces of an axis, the low one's neighbour and the high one's, at the exponents of
// the sum (I: of the pair, ep).
struct FxPair {
    i64 E, I, X, Y;
};
__host__ __device__ __forceinline__ FxPair fx_pair(const FxFlux& lo, const FxFlux& hi, int ep, int e,
                                                   unsigned ef)
{
    const unsigned dl = ef - lo.ef, dh = ef - hi.ef;
    const int xl = (int)(dl & 0xffffu), xh = (int)(dh & 0xffffu), yl = (int)(dl >> 16), yh = (int)(dh >> 16);
    return FxPair{ fx_down(lo.E, e - lo.e) - fx_down(hi.E, e - hi.e),
                   fx_down(lo.I, ep - lo.e) - fx_down(hi.I, ep - hi.e),
                   fx_down(lo.X, xl) - fx_down(hi.X, xh), fx_down(lo.Y, yl) - fx_down(hi.Y, yh) };
}

__host__ __device__ __forceinline__ FxPair fx_scale(const FxPair& p, Split r)
{
    return FxPair{ fx_product(p.E, r), fx_product(p.I, r), fx_product(p.X, r), fx_product(p.Y, r) };
}

// West and east.
__host__ __device__ __forceinline__ FxSum fx_sum1(const FxFlux& w, const FxFlux& e)
{
    FxSum s;
    s.e = s.ex = s.ey = w.e > e.e ? w.e : e.e;
    s.ef = fx_max2(w.ef, e.ef);
    const FxPair x = fx_pair(w, e, s.ex, s.e, s.ef);
    s.E = x.E; s.X = x.X; s.Y = x.Y; s.Ix = x.I; s.Iy = 0;
    return s;
}

// West and east, south and north.  fx: Level::fx, 2 and 3 scale the x and the y pair by rho.
__host__ __device__ __forceinline__ FxSum fx_sum2(const FxFlux& w, const FxFlux& e, const FxFlux& b,
                                                  const FxFlux& n, int fx, Split rho)
{
    FxSum s;
    s.ex = w.e > e.e ? w.e : e.e;
    s.ey = b.e > n.e ? b.e : n.e;
    s.e = s.ex > s.ey ? s.ex : s.ey;
    s.ef = fx_max2(fx_max2(w.ef, e.ef), fx_max2(b.ef, n.ef));
    FxPair x = fx_pair(w, e, s.ex, s.e, s.ef), y = fx_pair(b, n, s.ey, s.e, s.ef);
    if (fx == 2) x = fx_scale(x, rho);
    if (fx == 3) y = fx_scale(y, rho);
    s.E = x.E + y.E; s.X = x.X + y.X; s.Y = x.Y + y.Y; s.Ix = x.I; s.Iy = y.I;
    return s;
}

// v 2^(t - 58) + i 2^(e - 61) (biased exponents) in FP64, in units of the larger of the
// two where both are there.
__host__ __device__ __forceinline__ double fx_joined(i64 v, int t, i64 i, int e)
{
    const int ei = i == 0 ? 0 : e - 3, m = ei > t ? ei : t;
    return fx_double(fx_down(v, m - t) + fx_down(i, m - ei), m - 1023);
}

// The sums in FP64: N_E / cb, N_F / cbF.
__host__ __device__ __forceinline__ double fx_value_E(const FxSum& s) { return fx_double(s.E, s.e - 1023); }
__host__ __device__ __forceinline__ double fx_value_X(const FxSum& s)
{
    return fx_joined(s.X, (int)(s.ef & 0xffffu), s.Ix, s.ex);
}
__host__ __device__ __forceinline__ double fx_value_Y(const FxSum& s)
{
    return fx_joined(s.Y, (int)(s.ef >> 16), s.Iy, s.ey);
}

}  // namespace m1
