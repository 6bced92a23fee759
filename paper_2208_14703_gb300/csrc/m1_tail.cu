// The coarse end of a cycle in one launch.
//
// The FP64 levels of a few thousand cells and fewer take as long as their launches:
// a cycle runs about ten dependent kernels on each, 5 to 9 us apiece whatever their
// size (launch, work list, descriptor, rows from L2, one pass, drain), with the chip
// idle.  Here a cluster of thread blocks holds all levels of one instance from the
// first of at most kTailCells cells down in its shared memory, one thread per cell,
// and walks the whole sequence of coarse visits (Algorithm 4, V, W or F) with a
// cluster barrier (0.2 us) between operations.
// (The mixed path's FP32 levels: m1_tail32.cu.)
//
// What bounds it: the chain of one cell (neighbours 2.1k clocks, the limiter 0.5k, or
// 3.6k in a warp with a limited cell, the local solve 2.3k, the closure 1.5k), not its
// FP64 or integer issue.  Measured: the levels of 64^2 and below of a 1024^2 FP64 cycle
// 0.12 ms.
//
// Layout: a level's cells are split into equal ranges of consecutive cells, one
// range per block (small levels: fewer blocks).  What a cell's neighbours need,
// its iterate and closure, is stored by the thread that forms the iterate, so
// each closure is evaluated once; neighbours in another block's range are read
// through distributed shared memory.
#include <cooperative_groups.h>

#include "m1_cell.cuh"
#include "m1_strip64.cuh"
#include "m1_tail.h"

namespace cg = cooperative_groups;

namespace m1 {

namespace {

constexpr int kTailThreads = 512;

// One level in the cluster's shared memory: `blocks` ranges of `per` cells, the
// arrays of a range at byte offset `off` of its block, one after another.
struct TailGeo {
    int nx, n, per, blocks, off;
    unsigned mx, mper;             // ceil(2^32 / nx), ceil(2^32 / per): k / nx = k mx >> 32 for k < 2^16
};

__device__ __forceinline__ int row_of(const TailGeo& g, int k)
{
    return g.mx ? (int)__umulhi((unsigned)k, g.mx) : k;
}

// Arrays of a range of `per` cells: the iterates e0, e1, v and f (which first holds
// the restricted residual) and the local solve's coefficients (formed by the first
// step of a fresh visit), 32 bytes a cell each; the blocks of e0 (first of v) and e1
// without S, 56 each (64, with it, would put a warp's cells on a quarter of the banks); sigma;
// the four neighbours (side_code); the two S.
enum { ARR_E = 0, ARR_V = 2, ARR_F = 3, ARR_Q = 4, ARR_P = 5, ARR_SIG = 7, ARR_NB = 8, ARR_S = 9 };

// A block without its S.
struct TailBlock {
    int e;
    unsigned ef;
    i64 E, Fx, Fy, Axx, Axy, Ayy;
};
constexpr int kTailBytes = 5 * 32 + 2 * 56 + 16 + 16 + 2 * 8;

__device__ __forceinline__ int arr_at(int a, int per)
{
    return (a < ARR_P ? a * 32 : a < ARR_SIG ? 5 * 32 + (a - ARR_P) * 56
          : a < ARR_S ? 5 * 32 + 2 * 56 + (a - ARR_SIG) * 16
                      : 5 * 32 + 2 * 56 + 2 * 16 + (a - ARR_S) * 8) * per;
}

// What a level's pseudo-time steps share: dtau c b, dtau c^2 b (the sums' factors),
// A = 1 + dtau diag, C = 1 + dtau C_v, the limiter's scale.
struct TailStep {
    double cbE, cbF, A, C;
    ConeScale cone;
};

// A cell's block that could not be formed (m1_fx.cuh: not regular): its
// neighbours and itself take the FP64 form.
constexpr int kIrregular = 1 << 20;

struct Tail {
    const Level<double>* L;             // descriptors, [0] = the tail's first level
    const TailGeo* geo;
    const TailStep* step;
    unsigned char* smem;           // this block's arrays
    int rank;
    cg::cluster_group cl;

    // cell k of array a of level l, wherever it lies
    template <typename T>
    __device__ const T* at(int l, int a, int k) const
    {
        const TailGeo& g = geo[l];
        const int b = (int)__umulhi((unsigned)k, g.mper);
        const T* p = reinterpret_cast<const T*>(smem + g.off + arr_at(a, g.per)) +
                     (k - b * g.per);
        return b == rank ? p : cl.map_shared_rank(p, b);
    }
    // this block's own cell q of its range
    template <typename T>
    __device__ T* own(int l, int a, int q) const
    {
        const TailGeo& g = geo[l];
        return reinterpret_cast<T*>(smem + g.off + arr_at(a, g.per)) + q;
    }
    __device__ Sig2<double>* sig(int l, int q) const
    {
        const TailGeo& g = geo[l];
        return reinterpret_cast<Sig2<double>*>(smem + g.off + arr_at(ARR_SIG, g.per)) + q;
    }
    // a cell of array a with the wall rules of fetch()
    __device__ Cell4<double> fetch(int l, int a, int i, int j, int kind) const
    {
        const Ghost g = ghost_map(L[l], i, j);
        return ghost_apply(L[l], *at<Cell4<double>>(l, a, (int)g.k), g, kind);
    }
};

// A cell's neighbour across a wall of the stencil, packed: its index in its range
// (16 bits), the range's block (8), and the wall rule there + 1 (0: none).
__device__ __forceinline__ unsigned side_code(const Tail& t, int l, int k, int i, int j, int wall)
{
    const Level<double>& L = t.L[l];
    int kn, rule = -1;
    const bool inside = wall == WALL_W ? i > 0 : wall == WALL_E ? i + 1 < L.nx
                      : wall == WALL_S ? j > 0 : j + 1 < L.ny;
    if (inside) {
        kn = wall == WALL_W ? k - 1 : wall == WALL_E ? k + 1 : wall == WALL_S ? k - L.nx : k + L.nx;
    } else if (L.bc[wall] == BC_PERIODIC) {
        kn = wall == WALL_W ? k + L.nx - 1 : wall == WALL_E ? k - L.nx + 1
           : wall == WALL_S ? k + L.n - L.nx : k - L.n + L.nx;
    } else {
        kn = k;
        rule = L.bc[wall];
    }
    const int b = (int)__umulhi((unsigned)kn, t.geo[l].mper);
    return (unsigned)(kn - b * t.geo[l].per) | (unsigned)b << 16 | (unsigned)(rule + 1) << 24;
}

__device__ __forceinline__ void put_block(const Tail& t, int l, int buf, int q,
                                          const Cell4<double>& u)
{
    FxCell c{};
    if (!(t.L[l].fx && fx_stage_cell(t.L[l], u, c))) c.e = kIrregular;
    *t.own<TailBlock>(l, ARR_P + buf, q) = TailBlock{ c.e, c.ef, c.E, c.Fx, c.Fy, c.Axx, c.Axy, c.Ayy };
    *t.own<i64>(l, ARR_S + buf, q) = c.S;
}

// What the neighbour across `wall` gives (its flux towards this cell).
__device__ __forceinline__ FxFlux side64(const Tail& t, int l, int buf, unsigned code, int wall,
                                         int k)
{
    const Level<double>& L = t.L[l];
    const int rule = (int)(code >> 24) - 1;
    FxCell c;
    if (rule == BC_INFLOW) {
        const int j = L.dim == 2 ? row_of(t.geo[l], k) : 0, q = wall < 2 ? j : k - j * L.nx;
        const double* p = L.inflow + (size_t)(wall * 3) * L.prof_len;
        const Cell4<double> u = { p[q], p[L.prof_len + q], p[2 * L.prof_len + q], 0.0 };
        if (!fx_stage_cell(L, u, c)) c.e = kIrregular;
    } else {
        const TailBlock* p = t.own<TailBlock>(l, ARR_P + buf, (int)(code & 0xffffu));
        const i64* ps = t.own<i64>(l, ARR_S + buf, (int)(code & 0xffffu));
        const int b = (int)(code >> 16) & 0xff;
        if (b != t.rank) {
            p = t.cl.map_shared_rank(p, b);
            ps = t.cl.map_shared_rank(ps, b);
        }
        c = FxCell{ p->e, p->ef, p->E, p->Fx, p->Fy, p->Axx, p->Axy, p->Ayy, *ps };
        if (rule == BC_REFLECT) {
            if (wall < 2) c.Fx = -c.Fx;
            else c.Fy = -c.Fy;
            c.Axy = -c.Axy;
        }
    }
    const FxSide side = wall < 2 ? fx_side_x(c) : fx_side_y(c);
    return wall == WALL_W || wall == WALL_S ? fx_flux_of<false>(c, side)
                                            : fx_flux_of<true>(c, side);
}

// The cell's neighbour sums in FP64 throughout (a block nearby is irregular).
__device__ __noinline__ void general_sums64(const Tail& t, int l, int arr, int k, bool two_d,
                                            double& NE, double& NFx, double& NFy)
{
    const Level<double>& L = t.L[l];
    const int j = two_d ? row_of(t.geo[l], k) : 0, i = k - j * L.nx;
    Staged<double> s[4];
    for (int w = 0; w < (two_d ? 4 : 2); ++w) {
        const Cell4<double> c = t.fetch(l, arr, i + (w == 0 ? -1 : w == 1 ? 1 : 0),
                                        j + (w == 2 ? -1 : w == 3 ? 1 : 0), KIND_STATE);
        s[w].E = c.E; s[w].Fx = c.Fx; s[w].Fy = c.Fy; s[w].T = c.T;
        closure(c.E, c.Fx, c.Fy, L.ic2, s[w].Pxx, s[w].Pxy, s[w].Pyy);
    }
    if (!two_d) s[2] = s[3] = s[0];
    strip_neighbours(L, s[0], s[1], s[2], s[3], two_d, NE, NFx, NFy);
}

// The neighbour sums of Eq. (9): over the factors cb (E) and cbF (F) when fx, else
// whole, formed in FP64 throughout.
__device__ __forceinline__ void sums64(const Tail& t, int l, int arr, int buf, int k, int q,
                                       bool two_d, double& NE, double& NFx, double& NFy, bool& fx)
{
    const Level<double>& L = t.L[l];
    const uint4 nb = *t.own<uint4>(l, ARR_NB, q);
    const FxFlux w = side64(t, l, buf, nb.x, WALL_W, k), e = side64(t, l, buf, nb.y, WALL_E, k);
    FxSum s;
    if (two_d) {
        const FxFlux b = side64(t, l, buf, nb.z, WALL_S, k), n = side64(t, l, buf, nb.w, WALL_N, k);
        s = fx_sum2(w, e, b, n, L.fx, split62(L.rho));
    } else {
        s = fx_sum1(w, e);
    }
    if (s.e == kIrregular) {
        general_sums64(t, l, arr, k, two_d, NE, NFx, NFy);
        fx = false;
        return;
    }
    fx = true;
    NE = fx_value_E(s);
    NFx = fx_value_X(s);
    NFy = fx_value_Y(s);
}

__device__ __forceinline__ void arrive64(const Tail& t, int l, int q, const Cell4<double>& v,
                                         const Cell4<double>& r)
{
    *t.own<Cell4<double>>(l, ARR_V, q) = v;
    *t.own<Cell4<double>>(l, ARR_F, q) = r;
    put_block(t, l, 0, q, v);
}

// One field (0 to 3: E, Fx, Fy, T) of cell (i, j) of level l restricted from level
// l - 1 (k_restrict): of the iterate, in buffer c there, into v, or of the residual,
// in the other, into f.  The walls' rules as indices and signs; an inflow wall, rare,
// by the whole cell's rules.
__device__ __forceinline__ void restrict_field(const Tail& t, int l, int c, int q, int i, int j,
                                               bool resid, int field)
{
    const Level<double>& Lf = t.L[l - 1];
    const bool two_d = Lf.dim == 2;
    const int arr = resid ? ARR_E + 1 - c : ARR_E + c;
    const StencilAxis x = stencil_axis(2 * i, Lf.nx, Lf.bc[WALL_W]);
    const StencilAxis y = stencil_axis(2 * j, Lf.ny, Lf.bc[WALL_S]);
    double v[3][3];
    if (x.rule == BC_INFLOW || (two_d && y.rule == BC_INFLOW)) {
        for (int b = 0; b < 3; ++b)
            for (int a = 0; a < 3; ++a) {
                if (!two_d && b != 1) { v[b][a] = 0.0; continue; }
                const Cell4<double> s = t.fetch(l - 1, arr, 2 * i + a - 1, two_d ? 2 * j + b - 1 : 0,
                                                resid ? KIND_DIFF : KIND_STATE);
                v[b][a] = field == 0 ? s.E : field == 1 ? s.Fx : field == 2 ? s.Fy : s.T;
            }
    } else {
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if (!two_d && b != 1) continue;
            const int row = two_d ? y.k[b] * Lf.nx : 0;
#pragma unroll
            for (int a = 0; a < 3; ++a)
                v[b][a] = reinterpret_cast<const double*>(
                    t.at<Cell4<double>>(l - 1, arr, row + x.k[a]))[field];
        }
        if (two_d && field == 2 && y.rule == BC_REFLECT)
#pragma unroll
            for (int a = 0; a < 3; ++a) v[0][a] = -v[0][a];
        if (field == 1 && x.rule == BC_REFLECT)
#pragma unroll
            for (int b = 0; b < 3; ++b) v[b][0] = -v[b][0];
    }
    double s = 0.0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (!two_d && b != 1) continue;
        const double wy = two_d ? (b == 1 ? 0.5 : 0.25) : 1.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) s = fma(wy * (a == 1 ? 0.5 : 0.25), v[b][a], s);
    }
    reinterpret_cast<double*>(t.own<Cell4<double>>(l, resid ? ARR_F : ARR_V, q))[field] = s;
}

__device__ __forceinline__ void op_cell(const Tail& t, int op, int l, int cur, int ccur,
                                        int k, int q, const Pseudo<double>& ps, double theta_c,
                                        unsigned& fails, unsigned& damped)
{
    typedef Cell4<double> C;
    const Level<double>& L = t.L[l];
    const bool two_d = L.dim == 2;
    if (op == TAIL_PROLONG) {
        const int j = two_d ? row_of(t.geo[l], k) : 0, i = k - j * L.nx;
        const int ic = i >> 1, jc = two_d ? j >> 1 : 0, ox = i & 1, oy = two_d ? j & 1 : 0;
        const double wt = pow2_neg<double>(ox + oy);
        // the coarse cells past the high walls under the rules of differences
        const Level<double>& Lc = t.L[l + 1];
        const bool xo = ic + 1 == Lc.nx, yo = two_d && jc + 1 == Lc.ny;
        const int bx = Lc.bc[WALL_E], by = Lc.bc[WALL_N];
        const int xk = !xo ? ic + 1 : bx == BC_PERIODIC ? 0 : ic;
        const int yk = !yo ? jc + 1 : by == BC_PERIODIC ? 0 : jc;
        const int off = (ARR_V - ARR_E - ccur) * t.geo[l + 1].per;
        C cu[2][2], cv[2][2];
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                if (b > oy || a > ox) continue;
                const C* p = t.at<C>(l + 1, ARR_E + ccur, (b ? yk : jc) * Lc.nx + (a ? xk : ic));
                cu[b][a] = p[0];
                cv[b][a] = p[off];
            }
        C pe = { 0, 0, 0, 0 };
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                if (b > oy || a > ox) continue;
                const bool bo = b && yo, ao = a && xo;
                if ((bo && by == BC_INFLOW) || (ao && bx == BC_INFLOW)) continue;
                const C &m = cu[b][a], &n = cv[b][a];
                const double wx = ao && bx == BC_REFLECT ? -wt : wt, wy = bo && by == BC_REFLECT ? -wt : wt;
                pe.E += wt * (m.E - n.E); pe.Fx += wx * (m.Fx - n.Fx);
                pe.Fy += wy * (m.Fy - n.Fy); pe.T += wt * (m.T - n.T);
            }
        const C u = *t.own<C>(l, ARR_E + cur, q);
        C tg = { u.E + pe.E, u.Fx + pe.Fx, u.Fy + pe.Fy, u.T + pe.T };
        if (!admissible(tg, L.c)) {
            const double th = theta_c * fmin(1.0, max_admissible_step64(u, pe, L.c));
            tg = C{ u.E + th * pe.E, u.Fx + th * pe.Fx, u.Fy + th * pe.Fy, u.T + th * pe.T };
            ++damped;
        }
        *t.own<C>(l, ARR_E + cur, q) = tg;
        put_block(t, l, cur, q, tg);
        return;
    }
    double NE, NFx, NFy;
    bool fx;
    const int arr = op == TAIL_FIRST ? ARR_V : ARR_E + cur, buf = op == TAIL_FIRST ? 0 : cur;
    sums64(t, l, arr, buf, k, q, two_d, NE, NFx, NFy, fx);
    const C u = *t.own<C>(l, arr, q);
    C b = *t.own<C>(l, ARR_F, q);
    Coef co;
    if (op == TAIL_PSEUDO) {
        co = *t.own<Coef>(l, ARR_Q, q);
    } else {
        const Sig2<double> sg = *t.sig(l, q);
        const double ka = L.cdt * sg.sa, kt = L.cdt * (sg.sa + sg.ss);
        const double fE = fx ? L.cb : 1.0, fF = fx ? L.cbF : 1.0;
        const double T2 = u.T * u.T, src_e = ka * fma(-L.a_r, T2 * T2, u.E), dF = L.diag + kt;
        const C a = { fma(-fE, NE, fma(L.diag, u.E, src_e)), fma(-fF, NFx, dF * u.Fx),
                      fma(-fF, NFy, dF * u.Fy), fma(L.c_v, u.T, -src_e) };
        if (op == TAIL_RESID) {
            *t.own<C>(l, ARR_E + 1 - cur, q) = C{ b.E - a.E, b.Fx - a.Fx, b.Fy - a.Fy, b.T - a.T };
            return;
        }
        b = C{ a.E + b.E, a.Fx + b.Fx, a.Fy + b.Fy, a.T + b.T };
        *t.own<C>(l, ARR_F, q) = b;
        co = make_coef(1.0, ps.dtau, L.diag, ka, kt, L.a_r);
        *t.own<Coef>(l, ARR_Q, q) = co;
    }
    const TailStep& ts = t.step[l];
    const double cbE = fx ? ts.cbE : ps.dtau, cbF = fx ? ts.cbF : ps.dtau;
    const double tau = limited_step64(u, b, ps.dtau, ps.theta, ps.s, L.c, ts.cone);
    bool ok;
    const C o = local_solve64(co, ts.A, ts.C, L.a_r, fma(cbE, NE, fma(tau, b.E, u.E)),
                              fma(cbF, NFx, fma(tau, b.Fx, u.Fx)),
                              fma(cbF, NFy, fma(tau, b.Fy, u.Fy)), fma(tau, b.T, u.T), ok, u.T);
    if (!ok) ++fails;
    const int out = op == TAIL_FIRST ? 1 : 1 - cur;
    *t.own<C>(l, ARR_E + out, q) = o;
    put_block(t, l, out, q, o);
}

// Items are (instance, first tail level), one cluster each.
__global__ void __launch_bounds__(kTailThreads, 1) k_tail(const Level<double>* __restrict__ lv,
                                                          int cap, int nlev, WorkList wl,
                                                          Ctl* __restrict__ ctls,
                                                          const unsigned char* __restrict__ prog,
                                                          const int2* __restrict__ progs)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Level<double> Ls[kTailLevels];
    __shared__ TailGeo geo[kTailLevels];
    __shared__ TailStep steps[kTailLevels];
    cg::cluster_group cl = cg::this_cluster();
    const int nb = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int w0 = blockIdx.x / nb, ws = gridDim.x / nb;
    const int nw = *wl.count;
    Tail t{ Ls, geo, steps, smem, rank, cl };
    for (int w = w0; w < nw; w += ws) {
        const int2 it = wl.items[w];
        if (skip(ctls, it.x)) continue;            // the same for the whole cluster
        Ctl* ctl = ctls + it.x;
        const int first = it.y, nl = nlev - first;
        const Level<double>* src = lv + (size_t)first * cap + it.x;
        static_assert(sizeof(Level<double>) % 8 == 0 && sizeof(Level<double>) <= 32 * 8, "one word per lane");
        for (int l = threadIdx.x / 32; l < nl; l += kTailThreads / 32) {
            const unsigned long long* s =
                reinterpret_cast<const unsigned long long*>(src + (size_t)l * cap);
            if ((threadIdx.x & 31) < sizeof(Level<double>) / 8)
                reinterpret_cast<unsigned long long*>(&Ls[l])[threadIdx.x & 31] =
                    s[threadIdx.x & 31];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int off = 0;
            for (int l = 0; l < nl; ++l) {
                TailGeo g;
                g.nx = Ls[l].nx;
                g.n = Ls[l].n;
                g.per = tail_per(g.n, nb);
                g.blocks = (g.n + g.per - 1) / g.per;
                g.off = off;
                g.mx = g.nx > 1 ? (unsigned)((0x100000000ull + g.nx - 1) / g.nx) : 0u;
                g.mper = (unsigned)((0x100000000ull + g.per - 1) / g.per);
                geo[l] = g;
                off += kTailBytes * g.per;
            }
        }
        __syncthreads();
        const Pseudo<double> ps = pseudo_of<double>(ctl);
        if (threadIdx.x < nl) {
            const Level<double>& L = Ls[threadIdx.x];
            steps[threadIdx.x] = TailStep{ ps.dtau * L.cb, ps.dtau * L.cbF, fma(ps.dtau, L.diag, 1.0),
                                           fma(ps.dtau, L.c_v, 1.0), cone_scale(ps.s, L.ic) };
        }
        const double theta_c = ctl->theta_c;
        unsigned fails = 0, damped = 0;
        for (int l = 0; l < nl; ++l)
            for (int q = threadIdx.x; q < geo[l].per; q += kTailThreads) {
                const int k = rank * geo[l].per + q;
                if (k >= geo[l].n) break;
                *t.sig(l, q) = Ls[l].sig[k];
                const int j = Ls[l].dim == 2 ? row_of(geo[l], k) : 0, i = k - j * Ls[l].nx;
                uint4 nb = make_uint4(side_code(t, l, k, i, j, WALL_W), side_code(t, l, k, i, j, WALL_E),
                                      0u, 0u);
                if (Ls[l].dim == 2) {
                    nb.z = side_code(t, l, k, i, j, WALL_S);
                    nb.w = side_code(t, l, k, i, j, WALL_N);
                }
                *t.own<uint4>(l, ARR_NB, q) = nb;
                if (l == 0) arrive64(t, 0, q, Ls[0].v[k], Ls[0].r[k]);
            }
        unsigned curs = 0;                          // bit l: the buffer of level l's iterate
        const int2 pr = progs[first];
        bool was_multi = true;
        for (int p = 0; p <= pr.y; ++p) {
            const int code = p < pr.y ? prog[pr.x + p] : 0;
            const int op = code & 7, l = code >> 3;
            // the levels the operation reads or writes: l, and (restriction, prolongation)
            // one more; a single block works while all of them lie in block 0
            const int lo = p == pr.y ? 0 : (op == TAIL_RESTRICT ? l - 1 : l);
            const bool multi = geo[lo].blocks > 1;
            if (multi || was_multi) cl.sync();
            else if (rank == 0) __syncthreads();
            was_multi = multi;
            if (p == pr.y) break;
            const int cur = (curs >> l) & 1;
            const int ccur = op == TAIL_RESTRICT ? (curs >> (l - 1)) & 1
                           : op == TAIL_PROLONG ? (curs >> (l + 1)) & 1 : 0;
            const int base = rank * geo[l].per, end = min(geo[l].per, geo[l].n - base);
            if (op == TAIL_RESTRICT) {
                // eight threads a cell, a field of one of its two arrays each
                for (int x = threadIdx.x; x < 8 * end; x += kTailThreads) {
                    const int q = x >> 3, k = base + q;
                    const int j = Ls[l].dim == 2 ? row_of(geo[l], k) : 0;
                    restrict_field(t, l, ccur, q, k - j * geo[l].nx, j, x & 4, x & 3);
                }
                if (end > 0) __syncthreads();
                for (int q = threadIdx.x; q < end; q += kTailThreads)
                    put_block(t, l, 0, q, *t.own<Cell4<double>>(l, ARR_V, q));
                continue;
            }
            for (int q = threadIdx.x; q < end; q += kTailThreads)
                op_cell(t, op, l, cur, ccur, base + q, q, ps, theta_c, fails, damped);
            if (op == TAIL_FIRST) curs |= 1u << l;
            else if (op == TAIL_PSEUDO) curs ^= 1u << l;
        }
        // the result to global memory, into both buffers of the tail's first level (the
        // other instances of the level decide which one the prolongation reads)
        for (int q = threadIdx.x; q < geo[0].per; q += kTailThreads) {
            const int k = rank * geo[0].per + q;
            if (k >= geo[0].n) break;
            const Cell4<double> o = *t.own<Cell4<double>>(0, ARR_E + (curs & 1), q);
            Ls[0].u[0][k] = o;
            Ls[0].u[1][k] = o;
        }
        if (fails) atomicAdd(&ctl->newton_fail, fails);
        if (damped) atomicAdd(&ctl->damped, damped);
        cl.sync();                                  // before the next item's arrays
    }
    cl.sync();                                      // no block leaves while another reads it
}

}  // namespace

size_t tail_smem(int n0, int nb, int dim, int nlev)
{
    size_t s = 0;
    for (int l = 0; l < nlev; ++l) {
        s += (size_t)kTailBytes * tail_per(n0, nb);
        n0 /= dim == 2 ? 4 : 2;
    }
    return s;
}

cudaError_t tail_prepare()
{
    const cudaError_t e =
        cudaFuncSetAttribute(k_tail, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, kTailSmem);
}

cudaError_t launch_tail(const Level<double>* lv, int cap, int nlev, WorkList wl, Ctl* ctls,
                        const unsigned char* prog, const int2* progs, size_t smem, int blocks,
                        cudaStream_t s)
{
    const int most = kTailClusters * kTailBlocks / blocks;
    const int clusters = wl.capacity < most ? (wl.capacity > 0 ? wl.capacity : 1) : most;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * blocks);
    cfg.blockDim = dim3(kTailThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = blocks;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_tail, lv, cap, nlev, wl, ctls, prog, progs);
}

}  // namespace m1
