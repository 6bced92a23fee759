// The 3D operator in fixed point: m1_fx.cuh on three axes.
//
// A cell's block holds its exponent, E, F / c (three) and the closure's six entries
// as 64-bit significands relative to E (values m 2^(e - 60)).  Blocks are kept in
// memory as planes (one coalesced 8-byte load per entry and warp), written by the
// pass that forms the state, so that every closure is evaluated once and a sweep
// is one pass: its neighbour sums need no FP64 operation, and its update takes
// eleven where the FP64 form issues about 150.
#pragma once
#include "m1_3d.cuh"
#include "m1_strip64.cuh"

namespace m1 {

constexpr int kIrregular3 = 1 << 20;             // exponent of a cell no block can hold

// Planes of a block array of n cells: E, Fx, Fy, Fz, xx, xy, xz, yy, yz, zz, then
// the exponents.
struct Blocks3 {
    i64* m;
    int* e;
};

__host__ __device__ inline size_t blocks3_bytes(size_t n) { return n * (10 * sizeof(i64) + 4); }
__host__ __device__ inline Blocks3 blocks3_at(void* p, size_t n)
{
    return Blocks3{ static_cast<i64*>(p), reinterpret_cast<int*>(static_cast<i64*>(p) + 10 * n) };
}

struct FxCell3 {
    int e;
    i64 E, F[3], P[6];                           // xx, xy, xz, yy, yz, zz
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
    i64 mid = 0, F2 = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const u64 b = bits_of_double(F[a]);
        const int d = (int)te - (int)((unsigned)(b >> 52) & 0x7ffu);
        ok = ok && d >= 0;
        const i64 x = fx_align(b, d);
        s[a] = split62(x);
        o.F[a] = x >> 1;
        // partial sums of |F|^2 / 4 at scale 2^60: below 3 2^60 for any |F_a| < 2 E
        mid += madw(s[a].h, s[a].l, 0) >> 2;
        F2 += madw(s[a].h, s[a].h, 0) >> 2;
    }
    const Split sE = split62(xE);
    const i64 E2 = sqr62(sE);
    F2 += mid >> 30;                             // |F|^2 / 4
    ok = ok && F2 <= (E2 >> 2) + (E2 >> 12);
    i64 xi = E2 - 3 * F2;                        // x^2 - 3/4 |F|^2
    const i64 q2 = E2 >> 2;
    xi = xi > q2 ? xi : q2;
    i64 sg;
    const i64 D15 = fx_sigma_d(xE, xi, sg);
    const Split sD = split62(D15);
    constexpr i64 third = 768614336404564651ll;  // 2^61 / 3
    const i64 iso = mul62(split62((sg << 2) - xE), split62(third));
    int k = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const Split ga = split62(mul62(s[a], sD));
#pragma unroll
        for (int b = a; b < 3; ++b) o.P[k++] = mul62(ga, s[b], a == b ? iso : 0);
    }
    o.E = xE >> 1;
    o.e = (int)te - 1023;
    return ok;
}

__device__ __forceinline__ void put_block3(const G3& g, const EF& u, Blocks3 B, size_t n, size_t q)
{
    FxCell3 c;
    double F[3] = { u.F[0], u.F[1], u.F[2] };
    if (g.ic != 1.0)
        for (int a = 0; a < 3; ++a) F[a] *= g.ic;
    const bool ok = g.fx && fx_stage3(u.E, F, c);
    B.e[q] = ok ? c.e : kIrregular3;
    if (!ok) return;
    B.m[q] = c.E;
#pragma unroll
    for (int a = 0; a < 3; ++a) B.m[(1 + a) * n + q] = c.F[a];
#pragma unroll
    for (int a = 0; a < 6; ++a) B.m[(4 + a) * n + q] = c.P[a];
}

// Plane of the entry pairing axes d and a.
__device__ __forceinline__ constexpr int plane3(int d, int a)
{
    const int lo = d < a ? d : a, hi = d < a ? a : d;
    return 4 + (lo == 0 ? hi : lo == 1 ? 2 + hi : 5);
}

// A face of a cell: the neighbour's cell, the wall rule there (-1: none) and the
// exponent of its block.
struct Face3 {
    unsigned k;
    int rule, e;
};

// What the prescribed state of an inflow wall gives to the cell at p: e and, in m,
// E and F_a of its flux across axis d (side -1: E + F_d, F_a + P_da; +1: the
// differences).
static __device__ __noinline__ int inflow_flux3(const G3& g, int d, int side, const int p[3], i64 m[4])
{
    EF u;
    inflow_at(g, d, side < 0 ? 0 : 1, p, u);
    FxCell3 c;
    double F[3] = { u.F[0] * g.ic, u.F[1] * g.ic, u.F[2] * g.ic };
    const int e = g.fx && fx_stage3(u.E, F, c) ? c.e : kIrregular3;
    m[0] = side < 0 ? c.E + c.F[d] : c.E - c.F[d];
    for (int a = 0; a < 3; ++a) {
        const i64 P = c.P[plane3(d, a) - 4];
        m[1 + a] = side < 0 ? c.F[a] + P : c.F[a] - P;
    }
    return e;
}

template <int d, int side>
__device__ __forceinline__ Face3 face3(const G3& g, const Blocks3& B, unsigned q, const int p[3])
{
    const unsigned s = d == 0 ? 1u : d == 1 ? (unsigned)g.n[0] : (unsigned)g.n[0] * (unsigned)g.n[1];
    Face3 f = { side < 0 ? q - s : q + s, -1, 0 };
    if (side < 0 ? p[d] == 0 : p[d] + 1 == g.n[d]) {
        const int bc = g.bc[2 * d + (side < 0 ? 0 : 1)];
        if (bc == BC_PERIODIC) {
            f.k = side < 0 ? q + s * (unsigned)(g.n[d] - 1) : q - s * (unsigned)(g.n[d] - 1);
        } else {
            f.k = q;
            f.rule = bc;
            if (bc == BC_INFLOW) {
                i64 m[4];
                f.e = inflow_flux3(g, d, side, p, m);
                return f;
            }
        }
    }
    f.e = B.e[f.k];
    return f;
}

// Adds the flux across a face (with the wall rules of neighbour3), aligned to the
// exponent em of the sum: scale 2^(em - 57), three bits of headroom for six terms.
template <int d, int side>
__device__ __forceinline__ void add_face3(const G3& g, const Blocks3& B, size_t n, const Face3& f,
                                          const int p[3], int em, i64 sum[4])
{
    i64 m[4];
    if (f.rule == BC_INFLOW) {
        inflow_flux3(g, d, side, p, m);
    } else {
        const i64 sF = f.rule == BC_REFLECT ? -1 : 1;   // the wall-normal flux and P pairing it
        const i64 E = B.m[f.k];
        i64 F[3], P[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            F[a] = B.m[(1 + a) * n + f.k];
            P[a] = B.m[plane3(d, a) * n + f.k];
        }
        if (sF < 0) {
#pragma unroll
            for (int a = 0; a < 3; ++a)
                if (a == d) F[a] = -F[a];
                else P[a] = -P[a];
        }
        m[0] = side < 0 ? E + F[d] : E - F[d];
#pragma unroll
        for (int a = 0; a < 3; ++a) m[1 + a] = side < 0 ? F[a] + P[a] : F[a] - P[a];
    }
    // rounded down, or up on the high sides, as fx_to does
    const int sh = min(em - f.e + 3, 62);
    const i64 h = side < 0 ? 0 : (1ll << sh) - 1;
#pragma unroll
    for (int a = 0; a < 4; ++a) sum[a] += (m[a] + h) >> sh;
}

template <int d>
__device__ __forceinline__ void add_axis3(const G3& g, const Blocks3& B, size_t n, const Face3& lo,
                                          const Face3& hi, const int p[3], int em, i64 sum[4])
{
    if (g.rho[d] == 0) {
        add_face3<d, -1>(g, B, n, lo, p, em, sum);
        add_face3<d, 1>(g, B, n, hi, p, em, sum);
    } else {
        i64 x[4] = { 0, 0, 0, 0 };
        add_face3<d, -1>(g, B, n, lo, p, em, x);
        add_face3<d, 1>(g, B, n, hi, p, em, x);
#pragma unroll
        for (int a = 0; a < 4; ++a) sum[a] += fx_product(x[a], split62(g.rho[d]));
    }
}

// The neighbour sums N / (cb, cbF) of a cell; false when a block of the stencil is
// irregular.  The six exponents first, then one axis at a time.
__device__ __forceinline__ bool sums3(const G3& g, const Blocks3& B, size_t n, unsigned q,
                                      const int p[3], double N[4])
{
    const Face3 a0 = face3<0, -1>(g, B, q, p), a1 = face3<0, 1>(g, B, q, p);
    const Face3 b0 = face3<1, -1>(g, B, q, p), b1 = face3<1, 1>(g, B, q, p);
    const Face3 c0 = face3<2, -1>(g, B, q, p), c1 = face3<2, 1>(g, B, q, p);
    const int em = max(max(max(a0.e, a1.e), max(b0.e, b1.e)), max(c0.e, c1.e));
    if (em == kIrregular3) return false;
    i64 s[4] = { 0, 0, 0, 0 };
    add_axis3<0>(g, B, n, a0, a1, p, em, s);
    add_axis3<1>(g, B, n, b0, b1, p, em, s);
    add_axis3<2>(g, B, n, c0, c1, p, em, s);
#pragma unroll
    for (int a = 0; a < 4; ++a) N[a] = fx_double(s[a], em + 1);
    return true;
}

}  // namespace m1
