// The 3D operator in fixed point: m1_fx.cuh on three axes.
//
// A cell's block holds E, F / c (three) and the six entries of A as 64-bit significands at
// exponents of their own (FxCell's, on three axes), and S.  Blocks are kept in memory as planes (one coalesced 8-byte load per
// entry and warp), written by the pass that forms the state, so that every closure is
// evaluated once and a sweep is one pass: its neighbour sums need no FP64 operation, and its
// update takes eleven where the FP64 form issues about 150.
#pragma once
#include "m1_3d.cuh"
#include "m1_strip64.cuh"

namespace m1 {

constexpr unsigned kIrregular3 = 0x7fff;         // exponent of a cell no block can hold

// Biased exponents of E and Fx (halves of x), Fy and Fz (of y).
typedef uint2 Exp3;
__device__ __forceinline__ int exp3(const Exp3& t, int a)     // a: 0 E, 1 .. 3 F
{
    return (int)((a & 2 ? t.y : t.x) >> (a & 1 ? 16 : 0) & 0xffffu);
}

// Planes of a block array of n cells: E, Fx, Fy, Fz, xx, xy, xz, yy, yz, zz, S, then
// the exponents.
constexpr int kPlanes3 = 11;
struct Blocks3 {
    i64* m;
    Exp3* e;
};

__host__ __device__ inline size_t blocks3_bytes(size_t n) { return n * (kPlanes3 * sizeof(i64) + sizeof(Exp3)); }
__host__ __device__ inline Blocks3 blocks3_at(void* p, size_t n)
{
    return Blocks3{ static_cast<i64*>(p), reinterpret_cast<Exp3*>(static_cast<i64*>(p) + kPlanes3 * n) };
}

struct FxCell3 {
    Exp3 t;
    i64 E, F[3], A[6], S;                        // A: xx, xy, xz, yy, yz, zz
};

// The closure of Eq. (5) and the block of a cell (fx_stage with three flux
// components); F over c.
__device__ __forceinline__ bool fx_stage3(double E, const double F[3], FxCell3& o)
{
    const u64 be = bits_of_double(E);
    const unsigned te = (unsigned)(be >> 52);
    bool ok = te - kFxMinExp <= kFxMaxExp - kFxMinExp;
    const i64 xE = (i64)(((be & 0xfffffffffffffull) | 0x10000000000000ull) << 9);
    Split s[3];
    int t[3], d[3];
    i64 neg[3], F2 = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const u64 b = bits_of_double(F[a]);
        const i64 m = fx_flux(b, t[a], ok);
        d[a] = (int)te - t[a];
        ok = ok && d[a] >= 0;
        s[a] = split62(m);
        neg[a] = (i64)b >> 63;
        o.F[a] = ((m >> 3) ^ neg[a]) - neg[a];
        // |F|^2 / 4 at scale 2^60: below 3 2^60 for any |F_a| < 2 E
        F2 += fx_down(sqr62(s[a]), 2 * d[a] + 2);
    }
    const Split sE = split62(xE);
    const i64 E2 = sqr62(sE);
    ok = ok && F2 <= (E2 >> 2) + (E2 >> 12);
    i64 xi = E2 - 3 * F2;                        // x^2 - 3/4 |F|^2
    const i64 q2 = E2 >> 2;
    xi = xi > q2 ? xi : q2;
    const Split sD = split62(fx_d15(xE, xi, o.S));
    int k = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const Split ga = split62(mul62(s[a], sD));
#pragma unroll
        for (int b = a; b < 3; ++b, ++k) {
            const i64 v = mul62(ga, s[b], 2) >> 2, n = neg[a] ^ neg[b];
            o.A[k] = (v ^ n) - n;
        }
    }
    o.E = xE >> 3;
    o.t = make_uint2((te & 0x7ffu) | (unsigned)t[0] << 16, (unsigned)t[1] | (unsigned)t[2] << 16);
    return ok;
}

__device__ __forceinline__ void put_block3(const G3& g, const EF& u, Blocks3 B, size_t n, size_t q)
{
    FxCell3 c;
    double F[3] = { u.F[0], u.F[1], u.F[2] };
    if (g.ic != 1.0)
        for (int a = 0; a < 3; ++a) F[a] *= g.ic;
    const bool ok = g.fx && fx_stage3(u.E, F, c);
    B.e[q] = ok ? c.t : make_uint2(kIrregular3, 0);
    if (!ok) return;
    B.m[q] = c.E;
#pragma unroll
    for (int a = 0; a < 3; ++a) B.m[(1 + a) * n + q] = c.F[a];
#pragma unroll
    for (int a = 0; a < 6; ++a) B.m[(4 + a) * n + q] = c.A[a];
    B.m[10 * n + q] = c.S;
}

// Plane of the entry pairing axes d and a.
__device__ __forceinline__ constexpr int plane3(int d, int a)
{
    const int lo = d < a ? d : a, hi = d < a ? a : d;
    return 4 + (lo == 0 ? hi : lo == 1 ? 2 + hi : 5);
}

// A face of a cell: the neighbour's cell, the wall rule there (-1: none) and the
// exponents of its block.
struct Face3 {
    unsigned k;
    int rule;
    Exp3 t;
};

// What a cell gives across a face on axis d: m[0] E +- F_d and m[1 + a] F_a +- A_da, at its
// exponents and, from the high side, with the sign changed (FxFlux on three axes); and S.
struct Flux3 {
    i64 m[4], I;
};
template <int d, int side>
__device__ __forceinline__ Flux3 flux3(const Exp3& t, i64 E, const i64 F[3], const i64 A[3], i64 S)
{
    const int n = exp3(t, 0) - exp3(t, 1 + d);
    Flux3 o;
    o.I = S;
    o.m[0] = side < 0 ? fx_down(F[d], n) + E : fx_down(F[d], n) - E;
#pragma unroll
    for (int a = 0; a < 3; ++a) o.m[1 + a] = side < 0 ? fx_down(A[a], n) + F[a] : fx_down(A[a], n) - F[a];
    return o;
}

// That of the prescribed state of an inflow wall to the cell at p (side -1: the low wall),
// and the block's exponents.
template <int d, int side>
static __device__ __noinline__ Exp3 inflow_flux3(const G3& g, const int p[3], Flux3& o)
{
    EF u;
    inflow_at(g, d, side < 0 ? 0 : 1, p, u);
    FxCell3 c;
    double F[3] = { u.F[0] * g.ic, u.F[1] * g.ic, u.F[2] * g.ic };
    if (!(g.fx && fx_stage3(u.E, F, c))) return make_uint2(kIrregular3, 0);
    const i64 A[3] = { c.A[plane3(d, 0) - 4], c.A[plane3(d, 1) - 4], c.A[plane3(d, 2) - 4] };
    o = flux3<d, side>(c.t, c.E, c.F, A, c.S);
    return c.t;
}

template <int d, int side>
__device__ __forceinline__ Face3 face3(const G3& g, const Blocks3& B, unsigned q, const int p[3])
{
    const unsigned s = d == 0 ? 1u : d == 1 ? (unsigned)g.n[0] : (unsigned)g.n[0] * (unsigned)g.n[1];
    Face3 f = { side < 0 ? q - s : q + s, -1, make_uint2(0, 0) };
    if (side < 0 ? p[d] == 0 : p[d] + 1 == g.n[d]) {
        const int bc = g.bc[2 * d + (side < 0 ? 0 : 1)];
        if (bc == BC_PERIODIC) {
            f.k = side < 0 ? q + s * (unsigned)(g.n[d] - 1) : q - s * (unsigned)(g.n[d] - 1);
        } else {
            f.k = q;
            f.rule = bc;
            if (bc == BC_INFLOW) {
                Flux3 m;
                f.t = inflow_flux3<d, side>(g, p, m);
                return f;
            }
        }
    }
    f.t = B.e[f.k];
    return f;
}

// Adds the flux across a face (with the wall rules of neighbour3), aligned to the
// exponents tm of the sum (I: to ep); those from the high side are taken off.
template <int d, int side>
__device__ __forceinline__ void add_face3(const G3& g, const Blocks3& B, size_t n, const Face3& f,
                                          const int p[3], const Exp3& tm, int ep, i64 sum[4],
                                          i64& I)
{
    Flux3 m;
    if (f.rule == BC_INFLOW) {
        inflow_flux3<d, side>(g, p, m);
    } else {
        i64 F[3], A[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            F[a] = B.m[(1 + a) * n + f.k];
            A[a] = B.m[plane3(d, a) * n + f.k];
        }
        if (f.rule == BC_REFLECT) {                     // the wall-normal flux and A pairing it
#pragma unroll
            for (int a = 0; a < 3; ++a)
                if (a == d) F[a] = -F[a];
                else A[a] = -A[a];
        }
        m = flux3<d, side>(f.t, B.m[f.k], F, A, B.m[10 * n + f.k]);
    }
    const uint2 dt = make_uint2(tm.x - f.t.x, tm.y - f.t.y);
    const i64 i = fx_down(m.I, ep - exp3(f.t, 0));
    I = side < 0 ? I + i : I - i;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const i64 v = fx_down(m.m[a], exp3(dt, a));
        sum[a] = side < 0 ? sum[a] + v : sum[a] - v;
    }
}

template <int d>
__device__ __forceinline__ void add_axis3(const G3& g, const Blocks3& B, size_t n, const Face3& lo,
                                          const Face3& hi, const int p[3], const Exp3& tm, i64 sum[4],
                                          i64 I[3], int eI[3])
{
    const int ep = max(exp3(lo.t, 0), exp3(hi.t, 0));
    I[d] = 0;
    eI[d] = ep;
    if (g.rho[d] == 0) {
        add_face3<d, -1>(g, B, n, lo, p, tm, ep, sum, I[d]);
        add_face3<d, 1>(g, B, n, hi, p, tm, ep, sum, I[d]);
    } else {
        i64 x[4] = { 0, 0, 0, 0 };
        add_face3<d, -1>(g, B, n, lo, p, tm, ep, x, I[d]);
        add_face3<d, 1>(g, B, n, hi, p, tm, ep, x, I[d]);
        const Split rho = split62(g.rho[d]);
#pragma unroll
        for (int a = 0; a < 4; ++a) sum[a] += fx_product(x[a], rho);
        I[d] = fx_product(I[d], rho);
    }
}

// The neighbour sums N / (cb, cbF) of a cell; false when a block of the stencil is
// irregular.  The six faces' exponents first, then one axis at a time.
__device__ __forceinline__ bool sums3(const G3& g, const Blocks3& B, size_t n, unsigned q,
                                      const int p[3], double N[4])
{
    const Face3 a0 = face3<0, -1>(g, B, q, p), a1 = face3<0, 1>(g, B, q, p);
    const Face3 b0 = face3<1, -1>(g, B, q, p), b1 = face3<1, 1>(g, B, q, p);
    const Face3 c0 = face3<2, -1>(g, B, q, p), c1 = face3<2, 1>(g, B, q, p);
    auto most = [](const Exp3& a, const Exp3& b) { return make_uint2(fx_max2(a.x, b.x), fx_max2(a.y, b.y)); };
    const Exp3 tm = most(most(most(a0.t, a1.t), most(b0.t, b1.t)), most(c0.t, c1.t));
    if (exp3(tm, 0) == (int)kIrregular3) return false;
    i64 s[4] = { 0, 0, 0, 0 }, I[3];
    int eI[3];
    add_axis3<0>(g, B, n, a0, a1, p, tm, s, I, eI);
    add_axis3<1>(g, B, n, b0, b1, p, tm, s, I, eI);
    add_axis3<2>(g, B, n, c0, c1, p, tm, s, I, eI);
    N[0] = fx_double(s[0], exp3(tm, 0) - 1023);
#pragma unroll
    for (int a = 0; a < 3; ++a) N[1 + a] = fx_joined(s[1 + a], exp3(tm, 1 + a), I[a], eI[a]);
    return true;
}

}  // namespace m1
