// The FP64 strips in fixed point: the warp-strip march of m1_kernels.cu with the
// closure and the neighbour sums of Eq. (9) on the integer pipe (m1_fx.cuh), and
// the FP64 local solve with its iterations' corrections in FP32.
//
// What bounds them: the FP64 pipe (64 clocks a warp instruction and SM partition).
// A fine Jacobi update in FP64 alone issues 109 of them; here the closure (about 27,
// evaluated 1.2 times a cell) and the neighbour sums (26) take none, and the local
// solve 31 instead of 42.
#pragma once
#include "m1_fx.cuh"

namespace m1 {

__device__ __forceinline__ i64 shfl_i64(i64 v, int from)
{
    return __shfl_sync(0xffffffffu, v, from);
}

__device__ __forceinline__ FxFlux shfl_flux(const FxFlux& v, int from)
{
    FxFlux o;
    o.e = __shfl_sync(0xffffffffu, v.e, from);
    o.E = shfl_i64(v.E, from);
    o.Fx = shfl_i64(v.Fx, from);
    o.Fy = shfl_i64(v.Fy, from);
    return o;
}

// A flux at scale 2^(e - 58) of the exponent e >= v.e (two bits of headroom for
// the sum of four).
__device__ __forceinline__ FxFlux fx_to(const FxFlux& v, int e)
{
    const int n = e - v.e + 2;
    return FxFlux{ e, fx_sar(v.E, n), fx_sar(v.Fx, n), fx_sar(v.Fy, n) };
}

__device__ __forceinline__ FxFlux fx_add(const FxFlux& a, const FxFlux& b)
{
    return FxFlux{ a.e, a.E + b.E, a.Fx + b.Fx, a.Fy + b.Fy };
}

__device__ __forceinline__ FxFlux fx_scale(const FxFlux& a, Split r)
{
    return FxFlux{ a.e, mul62(split62(a.E), r), mul62(split62(a.Fx), r), mul62(split62(a.Fy), r) };
}

// What a cell gives across its faces: to the east and west, and (2D) to the north
// and south.
__device__ __forceinline__ FxFlux fx_east(const FxCell& c)
{
    return FxFlux{ c.e, c.E + c.Fx, c.Fx + c.Pxx, c.Fy + c.Pxy };
}
__device__ __forceinline__ FxFlux fx_west(const FxCell& c)
{
    return FxFlux{ c.e, c.E - c.Fx, c.Fx - c.Pxx, c.Fy - c.Pxy };
}
__device__ __forceinline__ FxFlux fx_north(const FxCell& c)
{
    return FxFlux{ c.e, c.E + c.Fy, c.Fx + c.Pxy, c.Fy + c.Pyy };
}
__device__ __forceinline__ FxFlux fx_south(const FxCell& c)
{
    return FxFlux{ c.e, c.E - c.Fy, c.Fx - c.Pxy, c.Fy - c.Pyy };
}

__device__ __forceinline__ bool fx_stage_cell(const Level<double>& L, const Cell4<double>& c,
                                              FxCell& o)
{
    double Fx = c.Fx, Fy = c.Fy;
    if (L.ic != 1.0) { Fx *= L.ic; Fy *= L.ic; }
    return fx_stage(c.E, Fx, Fy, o);
}

// The strip march of strip_march in fixed point: calls cell(k, p, s) for each own
// cell, s the sum of its neighbours' fluxes (N_E = cb s.E 2^(s.e - 58), N_F with
// cbF) and p = pre(k), loaded one row ahead.  Returns false, for the whole warp,
// when some staged cell was not regular: every result of the strip is then to be
// formed again by the FP64 form.
template <typename Pre, typename Cell>
__device__ __forceinline__ bool strip_march_fx(const Level<double>& L, int2 it, int lane,
                                               const Cell4<double>* __restrict__ src, Pre&& pre,
                                               Cell&& cell)
{
    const int nx = L.nx, ny = L.ny;
    const bool two_d = L.dim == 2;
    const int x0 = (it.y % L.sx) * kStripW, y0 = (it.y / L.sx) * L.sh;
    const int i = min(x0 - 1 + lane, nx);
    const bool colfast = x0 >= 1 && x0 + kStripW + 1 <= nx;
    const bool own = lane >= 1 && lane <= kStripW && i < nx;
    const int rows = min(L.sh, ny - y0);
    auto load = [&](int j) {
        return colfast && j >= 0 && j < ny ? src[(size_t)j * nx + i] : fetch(L, src, i, j, KIND_STATE);
    };
    bool ok = true;
    Cell4<double> rn{};
    FxCell cur, next;
    FxFlux below{};                              // what row j - 1 gives to row j
    size_t k = (size_t)y0 * nx + i;
    decltype(pre(k)) pn{};
    if (own) pn = pre(k);
    const Cell4<double> r0 = load(y0);
    if (two_d) {
        const Cell4<double> rb = load(y0 - 1);
        rn = load(y0 + 1);
        ok = fx_stage_cell(L, rb, next) && ok;
        below = fx_north(next);
    }
    ok = fx_stage_cell(L, r0, cur) && ok;
    const Split rho = split62(L.rho);
#pragma unroll 1
    for (int r = 0; r < rows; ++r, k += nx) {
        if (two_d) {
            ok = fx_stage_cell(L, rn, next) && ok;
            if (r + 1 < rows) rn = load(y0 + r + 2);
        }
        const auto p = pn;
        if (own && r + 1 < rows) pn = pre(k + nx);
        const FxFlux w = shfl_flux(fx_east(cur), (lane + 31) & 31);
        const FxFlux e = shfl_flux(fx_west(cur), (lane + 1) & 31);
        int em = max(w.e, e.e);
        FxFlux s;
        if (two_d) {
            const FxFlux n = fx_south(next);
            em = max(em, max(below.e, n.e));
            s = fx_add(fx_to(w, em), fx_to(e, em));
            FxFlux sy = fx_add(fx_to(below, em), fx_to(n, em));
            if (L.fx == 2) s = fx_scale(s, rho);
            if (L.fx == 3) sy = fx_scale(sy, rho);
            s = fx_add(s, sy);
            below = fx_north(cur);
            if (own) cell(k, p, s);
            cur = next;
        } else {
            s = fx_add(fx_to(w, em), fx_to(e, em));
            if (own) cell(k, p, s);
        }
    }
    return __all_sync(0xffffffffu, ok);
}

// x rounded toward zero to FP32: values below its normal range give 0, above it
// (and NaN) infinity.  For corrections that need a few digits.
__device__ __forceinline__ float narrow_rz(double x, int eshift = 0)
{
    const int hi = __double2hiint(x);
    const int mag = (hi & 0x7fffffff) - (eshift << 20);        // x 2^-eshift
    unsigned f = __funnelshift_l((unsigned)__double2loint(x), (unsigned)mag, 3) - (896u << 23);
    f = mag < (897 << 20) ? 0u : (mag >= (1151 << 20) ? 0x7f800000u : f);
    return __uint_as_float(f | ((unsigned)hi & 0x80000000u));
}

// (double)x for a normal FP32 x; zero gives a number below 2^-126.
__device__ __forceinline__ double widen_normal(float x)
{
    const unsigned u = __float_as_uint(x);
    return __hiloint2double((int)((((u & 0x7fffffffu) >> 3) + (896u << 20)) | (u & 0x80000000u)),
                            (int)(u << 29));
}

// The root of C T + K T^4 = R in FP64: Newton in FP32 to about 2e-7, then two
// Newton corrections whose residuals are formed in FP64 and whose quotients in
// FP32 (each correction needs only the digits it adds: the first leaves an error
// near 1e-13, the second FP64 rounding).  Ten FP64 operations; a Halley step with
// an FP64 quotient took 17.  Where FP32 cannot seed the root, Quartic<double>
// takes the cell.
__device__ __forceinline__ double quartic64(double C, double K, double R, bool& ok)
{
    const float Cf = narrow_rz(C), Kf = narrow_rz(K), Rf = narrow_rz(R);
    const float K4 = 4.0f * Kf;
    float T = fminf(Rf * seed_rcp(Cf), Fm<float>::sqrt(Fm<float>::sqrt(Rf * seed_rcp(Kf))));
    bool conv = false;
    for (int it = 0; it < 40; ++it) {
        const float T3 = T * T * T;
        const float g = fmaf(Kf, T3 * T, Cf * T) - Rf;
        const float dT = g * seed_rcp(fmaf(K4, T3, Cf));
        T -= dT;
        // Newton's error is at most 1.5 dT^2 / T here (g'' T <= 3 g')
        if (fabsf(dT) <= 3e-4f * T) { conv = true; break; }
    }
    const int eR = (int)((__float_as_uint(Rf) >> 23) & 0xffu) - 127;
    // 1 / g' in units of 1 / R: at most about 2 T, so the quotients below stay in range
    const float q = seed_rcp(fmaf(K4, T * T * T, Cf)) * __uint_as_float((unsigned)(eR + 127) << 23);
    if (conv && T > 1e-18f && T < 1e18f && q > 1e-18f * T && eR > -126) {
        double Td = widen_normal(T);
        double T2 = Td * Td, KT2 = K * T2;
        const float d1 = narrow_rz(fma(KT2, T2, fma(C, Td, -R)), eR) * q;
        Td -= widen_normal(d1);
        T2 = Td * Td;
        KT2 = K * T2;
        const float d2 = narrow_rz(fma(KT2, T2, fma(C, Td, -R)), eR) * q;
        if (fabsf(d1) <= 1e-5f * T && fabsf(d2) <= 1e-9f * T) {
            ok = true;
            return Td - widen_normal(d2);
        }
    }
    return Quartic<double>::solve(C, K, R, ok);
}

// local_solve in FP64 for the strips: quartic64, and without absorption the
// quotients by one shared reciprocal (each followed by its remainder's
// correction) instead of FP64 divisions.
__device__ __forceinline__ Cell4<double> local_solve64(double w0, double w1, double diag, double ka,
                                                       double kt, double c_v, double a_r, double bE,
                                                       double bFx, double bFy, double bT, bool& ok)
{
    Cell4<double> o;
    const double A = fma(w1, diag, w0), k = w1 * ka, C = fma(w1, c_v, w0);
    const double dF = fma(w1, diag + kt, w0);
    ok = true;
    if (is_zero_f64(k)) {
        const double ip = Fm<double>::rcp(dF * A), iF = A * ip, iA = dF * ip;
        o.Fx = bFx * iF;
        o.Fy = bFy * iF;
        const double q = bE * iA;
        o.E = fma(fma(-A, q, bE), iA, q);
        o.T = bT;
        if (C != 1.0) o.T = bT / C;
        return o;
    }
    const double dE = A + k;
    const double ip = Fm<double>::rcp(dF * dE);
    const double iF = dE * ip, iAk = dF * ip;
    o.Fx = bFx * iF;
    o.Fy = bFy * iF;
    const double ark = a_r * (k * iAk);
    const double T = quartic64(C, A * ark, fma(k * iAk, bE, bT), ok);
    const double T2 = T * T;
    o.T = T;
    o.E = fma(ark, T2 * T2, bE * iAk);
    return o;
}

}  // namespace m1
