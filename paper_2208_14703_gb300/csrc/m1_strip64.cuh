// The FP64 strips in fixed point: the warp-strip march of m1_kernels.cu with the
// closure and the neighbour sums of Eq. (9) on the integer pipe (m1_fx.cuh), and
// the FP64 local solve with its iterations' corrections in FP32.
//
// What bounds them: the FP64 pipe (64 clocks a warp instruction and SM partition).
// A fine Jacobi update in FP64 alone issues 109 of them; here the closure (about 27,
// evaluated 1.2 times a cell) and the neighbour sums (26) take none, and the local
// solve seven instead of 42: its coefficients depend on the opacities and the time
// step alone (kept per cell over a step on the fine level), and its quartic is
// solved in fixed point.
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
    o.ef = __shfl_sync(0xffffffffu, v.ef, from);
    o.E = shfl_i64(v.E, from);
    o.I = shfl_i64(v.I, from);
    o.X = shfl_i64(v.X, from);
    o.Y = shfl_i64(v.Y, from);
    return o;
}

__device__ __forceinline__ bool fx_stage_cell(const Level<double>& L, const Cell4<double>& c,
                                              FxCell& o)
{
    double Fx = c.Fx, Fy = c.Fy;
    if (L.ic != 1.0) { Fx *= L.ic; Fy *= L.ic; }
    return fx_stage(c.E, Fx, Fy, o);
}

// The strip march of strip_march in fixed point: calls cell(k, p, s) for each own
// cell, s the sum of its neighbours' fluxes (N_E = cb fx_value_E(s), N_F with cbF)
// and p = pre(k), loaded one row ahead.  Returns false, for the whole warp,
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
        below = fx_flux_of<false>(next, fx_side_y(next));
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
        const FxSide side = fx_side_x(cur);
        const FxFlux w = shfl_flux(fx_flux_of<false>(cur, side), (lane + 31) & 31);
        const FxFlux e = shfl_flux(fx_flux_of<true>(cur, side), (lane + 1) & 31);
        if (two_d) {
            const FxFlux n = fx_flux_of<true>(next, fx_side_y(next));
            const FxSum s = fx_sum2(w, e, below, n, L.fx, rho);
            below = fx_flux_of<false>(cur, fx_side_y(cur));
            if (own) cell(k, p, s);
            cur = next;
        } else {
            const FxSum s = fx_sum1(w, e);
            if (own) cell(k, p, s);
        }
    }
    return __all_sync(0xffffffffu, ok);
}

// The coefficients of one cell's local solve D^{-1} (local_solve in m1_device.cuh):
// with A = w0 + w1 diag and k = w1 ka, 1 / (w0 + w1 (diag + kt)), k / (A + k),
// 1 / (A + k) and K = a_r A k / (A + k).  (w0, w1) as there: (0, 1) for a Jacobi
// sweep, (1, dtau) for a pseudo-time step.
struct Coef {
    double iF, kk, iAk, K;
};

__device__ __forceinline__ Coef make_coef(double w0, double w1, double diag, double ka, double kt,
                                          double a_r)
{
    const double A = fma(w1, diag, w0), k = w1 * ka;
    const double dF = fma(w1, diag + kt, w0), dE = A + k;
    // one reciprocal serves both denominators: 1/a = b / (a b), 1/b = a / (a b)
    const double ip = Fm<double>::rcp(dF * dE);
    const double iAk = dF * ip, kk = k * iAk;
    return Coef{ dE * ip, kk, iAk, A * (a_r * kk) };
}

// The local solve with its coefficients given: seven FP64 operations, the quartic
// in fixed point (fx_quartic) or, where that cannot hold it, by Quartic<double>.
// A is used without absorption only: E = bE / A with the quotient's remainder added.
// Tseed: a temperature near the solution (0: none).
__device__ __forceinline__ Cell4<double> local_solve64(const Coef& q, double A, double C, double a_r,
                                                       double bE, double bFx, double bFy, double bT,
                                                       bool& ok, double Tseed = 0.0)
{
    Cell4<double> o;
    ok = true;
    o.Fx = bFx * q.iF;
    o.Fy = bFy * q.iF;
    if (is_zero_f64(q.kk)) {
        const double e = bE * q.iAk;
        o.E = fma(fma(-A, e, bE), q.iAk, e);
        o.T = bT;
        if (C != 1.0) o.T = bT / C;
        return o;
    }
    const double R = fma(q.kk, bE, bT);
    double T4;
    if (!fx_quartic(C, q.K, R, o.T, T4, narrow_rz(Tseed))) {
        o.T = Quartic<double>::solve(C, q.K, R, ok);
        const double T2 = o.T * o.T;
        T4 = T2 * T2;
    }
    double ark = q.kk;
    if (a_r != 1.0) ark *= a_r;
    o.E = fma(ark, T4, bE * q.iAk);
    return o;
}

// x / y and sqrt(x) for the limited step, by the refined estimates of Fm<double>
// where both arguments are of ordinary size, else IEEE.
__device__ __forceinline__ bool ordinary(double x)
{
    return ((unsigned)(__double2hiint(x) >> 20) & 0x7ffu) - 200u < 1647u;
}
__device__ __forceinline__ double quotient(double x, double y)
{
    if (!ordinary(y)) return x / y;
    const double r = Fm<double>::rcp(y), q = x * r;
    return fma(fma(-y, q, x), r, q);
}

// max_admissible_step in thirty FP64 operations at most where the IEEE divisions and
// square root took sixty-five; the same bounds, each within an ulp or two.
__device__ __forceinline__ double cone_step(double a, double b, double c0)
{
    c0 = c0 > 0.0 ? 0.0 : c0;
    const double disc = fma(b, b, -(a * c0));
    const double sd = disc > 0.0 && ordinary(disc) ? Fm<double>::sqrt(disc) : sqrt(disc);
    if (a > 0.0) return b <= 0.0 ? quotient(sd - b, a) : quotient(-c0, b + sd);
    if (a < 0.0) return b > 0.0 && disc >= 0.0 ? quotient(-c0, b + sd) : (double)INFINITY;
    return b > 0.0 ? quotient(-c0, 2.0 * b) : (double)INFINITY;
}

// A bound u / (-d) on tau where d < 0.
__device__ __forceinline__ double plane_step(double u, double d)
{
    return d < 0.0 ? quotient(-u, d) : (double)INFINITY;
}

__device__ __forceinline__ double max_admissible_step64(const Cell4<double>& u,
                                                        const Cell4<double>& d, double c)
{
    const double c2 = c * c, cd = c2 * d.E, cu = c2 * u.E;
    const double a = fma(-cd, d.E, fma(d.Fy, d.Fy, d.Fx * d.Fx));
    const double b = fma(-cu, d.E, fma(u.Fy, d.Fy, u.Fx * d.Fx));
    const double c0 = fma(-cu, u.E, fma(u.Fy, u.Fy, u.Fx * u.Fx));
    return fmin(fmin(plane_step(u.E, d.E), plane_step(u.T, d.T)), cone_step(a, b, c0));
}

// Whether u + s f is admissible, decided in FP32 where that is beyond doubt (values
// rounded toward zero, a margin of 1e-6 of the terms' sizes where the roundings
// leave at most 6e-7): 1 yes, -1 no, 0 unknown.
//
// The question is put to E, T and F / c, so that light speeds of any unit system leave
// squares of the size of E^2 (with |F| against c E, CGS light speeds passed FP32's range
// at E = 6e8).  It is answered inside these bounds, where nothing that FP32 flushes to
// zero or overflows can reach a margin: s and 1 / c within 1e-30 .. 1e15, their product
// at most 1e15 (what narrow_rz drops, 1.2e-38, stays below 1e-22), E and T above 1e-15,
// E below 1e15, the sum of squares within 1e-30 .. 1e37 of an answer that rests on it.
struct ConeScale {
    float s, ic;                   // s and 1 / c; s NaN where they are out of range
};

__host__ __device__ __forceinline__ ConeScale cone_scale(double s, double ic)
{
    const float s32 = (float)s, i32 = (float)ic;
    const bool ok = s32 >= 1e-30f && s32 <= 1e15f && i32 >= 1e-30f && i32 <= 1e15f &&
                    s32 * i32 <= 1e15f;
    return ConeScale{ ok ? s32 : float_of_bits(0x7fc00000u), i32 };
}

struct FluxSum {
    ConeScale q;
    float hi = 0.f, lo = 0.f;      // squared length of (u + s f) / c, margins added, taken off
    __host__ __device__ __forceinline__ explicit FluxSum(const ConeScale& scale) : q(scale) {}
    __host__ __device__ __forceinline__ void add(double u64, double f64)
    {
        const float u = q.ic * narrow_rz(u64), f = q.ic * (q.s * narrow_rz(f64));
        const float p = fabsf(u + f), m = 1e-6f * (fabsf(u) + fabsf(f));
        hi = fmaf(p + m, p + m, hi);
        lo = fmaf(fmaxf(p - m, 0.f), fmaxf(p - m, 0.f), lo);
    }
};

__host__ __device__ __forceinline__ int admissible_sure(double E, double T, double dE, double dT,
                                                        const FluxSum& F)
{
    const float m = 1e-6f;
    const float uE = narrow_rz(E), uT = narrow_rz(T);
    if (!(uE > 1e-15f && uT > 1e-15f && uE < 1e15f)) return 0;
    const float fE = F.q.s * narrow_rz(dE), fT = F.q.s * narrow_rz(dT);
    const float mE = m * (uE + fabsf(fE)), mT = m * (uT + fabsf(fT));
    const float pE = uE + fE, pT = uT + fT;
    if (pE < -mE || pT < -mT) return -1;
    const float lo = pE - mE, hi = pE + mE;
    if (pT > mT && lo > 1e-15f && F.hi <= 0.99999f * lo * lo && F.hi < 1e37f) return 1;
    if (F.lo >= 1.00001f * hi * hi && F.lo > 1e-30f && F.lo < 1e37f) return -1;
    return 0;
}

// limited_step with the question whether it binds put in FP32 first.
__device__ __forceinline__ double limited_step64(const Cell4<double>& u, const Cell4<double>& f,
                                                 double dtau, double theta, double s, double c,
                                                 const ConeScale& q)
{
    FluxSum F(q);
    F.add(u.Fx, f.Fx);
    F.add(u.Fy, f.Fy);
    const int sure = admissible_sure(u.E, u.T, f.E, f.T, F);
    if (sure > 0) return dtau;
    if (sure == 0) {
        const Cell4<double> p = { fma(s, f.E, u.E), fma(s, f.Fx, u.Fx), fma(s, f.Fy, u.Fy),
                                  fma(s, f.T, u.T) };
        if (admissible_c2<double, false>(p, c * c)) return dtau;
    }
    return fmin(dtau, theta * max_admissible_step64(u, f, c));
}

}  // namespace m1
