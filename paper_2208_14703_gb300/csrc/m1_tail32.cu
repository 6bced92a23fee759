// The coarse end of a mixed cycle in one launch: m1_tail.cu for the FP32 hierarchy in
// correction form, on the functions of the strip kernels (m1_exact32.cuh), so that a level
// gives the same bits here and in launches of its own.
//
// A cluster of `blocks` thread blocks per instance, one thread per cell; between
// operations a cluster barrier.  What bounds an operation is the chain of dependent
// instructions of one cell (its neighbours' reads, the limited step, the Newton loop,
// the closure: about 2 us) and, at 1024 cells a block, instruction issue (4 us).  The
// transfers split a cell's arrays over three threads and take the walls' rules as index
// and sign choices: one thread a cell with a call per wall cell held the whole cluster up
// (12k to 18k clocks a restriction, now 4k to 12k).
// Measured: the five coarse levels of a 1024^2 mixed cycle (128^2 down to 8^2, 45
// operations) 0.115 ms; the cycle 0.685 ms with a launch for each, 0.575 ms so.  Eight
// served 256^2 to 1024^2 streams: 641 to 529 ms.  A batch of 24 of 64^2 to 512^2 (clusters of
// 4 blocks, tails from 64^2 down): no difference beyond the noise of 1%.
#include <cooperative_groups.h>

#include "m1_cell.cuh"
#include "m1_exact32.cuh"
#include "m1_tail.h"

namespace cg = cooperative_groups;

namespace m1 {

namespace {

typedef Cell4<float> C4;

constexpr int kThreads32 = 512;

struct Geo32 {
    int nx, n, per, blocks, off;
    unsigned mx, mper;             // ceil(2^32 / nx), ceil(2^32 / per)
};

// Arrays of a range of `per` cells, 16 bytes a cell each: iterates e0 (first P(w)), e1;
// closure differences P0, P1 (P1 first those of the FAS right-hand side); v, w, A(w),
// f (first the restricted residual); then sigma, 8.
enum { E0 = 0, P0 = 2, V = 4, W = 5, AW = 6, F = 7, SIG = 8 };
constexpr int kBytes32 = 8 * 16 + 8;

struct Tail32 {
    const Level<float>* L;
    const Geo32* geo;
    unsigned char* smem;
    int rank;
    unsigned ring;                 // bit l: level l's sweeps are the cp.async strips' (sums_x)
    cg::cluster_group cl;

    __device__ __forceinline__ const C4* at(int l, int a, int k) const
    {
        const Geo32& g = geo[l];
        const int b = (int)__umulhi((unsigned)k, g.mper);
        const C4* p = reinterpret_cast<const C4*>(smem + g.off + a * 16 * g.per) + (k - b * g.per);
        return b == rank ? p : cl.map_shared_rank(p, b);
    }
    __device__ __forceinline__ C4* own(int l, int a, int q) const
    {
        const Geo32& g = geo[l];
        return reinterpret_cast<C4*>(smem + g.off + a * 16 * g.per) + q;
    }
    __device__ __forceinline__ Sig2<float>* sig(int l, int q) const
    {
        const Geo32& g = geo[l];
        return reinterpret_cast<Sig2<float>*>(smem + g.off + SIG * 16 * g.per) + q;
    }
};

__device__ __forceinline__ int row32(const Geo32& g, int k)
{
    return g.mx ? (int)__umulhi((unsigned)k, g.mx) : k;
}

// A neighbour outside the grid, or w's at an inflow wall: rare, out of line.
__device__ __noinline__ Staged<float> wall32(const Tail32& t, int l, int ae, int ap, int wall, bool base,
                                      int k, int i, int j)
{
    const Level<float>& L = t.L[l];
    const int bc = L.bc[wall];
    if (bc == BC_INFLOW) {
        if (!base) return Staged<float>{};
        const int q = wall < 2 ? j : i;
        const float* p = L.inflow + (size_t)(wall * 3) * L.prof_len;
        Staged<float> s;
        s.E = p[q]; s.Fx = p[L.prof_len + q]; s.Fy = p[2 * L.prof_len + q];
        closure(s.E, s.Fx, s.Fy, L.ic2, s.Pxx, s.Pxy, s.Pyy);
        return s;
    }
    if (bc == BC_PERIODIC)
        k = wall == WALL_W ? k + L.nx - 1 : wall == WALL_E ? k - L.nx + 1
          : wall == WALL_S ? k + L.n - L.nx : k - L.n + L.nx;
    const C4 e = *t.at(l, ae, k), p = *t.at(l, ap, k);
    Staged<float> s = { e.E, e.Fx, e.Fy, p.E, p.Fx, p.Fy, 0.f };
    if (bc == BC_REFLECT) {
        if (wall < 2) s.Fx = -s.Fx;
        else s.Fy = -s.Fy;
        s.Pxy = -s.Pxy;
    }
    return s;
}

template <int WALL>
__device__ __forceinline__ Staged<float> side32(const Tail32& t, int l, int ae, int ap, bool base, int k,
                                         int q, int i, int j)
{
    const Level<float>& L = t.L[l];
    const bool inside = WALL == WALL_W ? i > 0 : WALL == WALL_E ? i + 1 < L.nx
                      : WALL == WALL_S ? j > 0 : j + 1 < L.ny;
    if (!inside) return wall32(t, l, ae, ap, WALL, base, k, i, j);
    const int s = WALL == WALL_W ? -1 : WALL == WALL_E ? 1 : WALL == WALL_S ? -L.nx : L.nx;
    const bool here = (unsigned)(q + s) < (unsigned)t.geo[l].per;
    const C4* pe = here ? t.own(l, ae, q + s) : t.at(l, ae, k + s);
    const C4* pp = here ? t.own(l, ap, q + s) : t.at(l, ap, k + s);
    const C4 e = *pe, p = *pp;
    return Staged<float>{ e.E, e.Fx, e.Fy, p.E, p.Fx, p.Fy, 0.f };
}

__device__ __forceinline__ Sums32 sums32(const Tail32& t, int l, int ae, int ap, bool base, bool xfused,
                                         int k, int q, int i, int j)
{
    const Level<float>& L = t.L[l];
    const Staged<float> w = side32<WALL_W>(t, l, ae, ap, base, k, q, i, j);
    const Staged<float> e = side32<WALL_E>(t, l, ae, ap, base, k, q, i, j);
    Staged<float> s{}, n{};
    if (L.dim == 2) {
        s = side32<WALL_S>(t, l, ae, ap, base, k, q, i, j);
        n = side32<WALL_N>(t, l, ae, ap, base, k, q, i, j);
    }
    Sums32 N;
    sums_x(L.c, L.bx, L.by, L.dim == 2, xfused, w, e, s, n, N.E, N.Fx, N.Fy);
    return N;
}

template <bool FAS>
__device__ __forceinline__ C4 closure32(const Level<float>& L, const C4& w, const C4& e)
{
    C4 p;
    closure_delta_x<FAS>(w.E, w.Fx, w.Fy, e.E, e.Fx, e.Fy, L.ic2, p.E, p.Fx, p.Fy);
    p.T = 0.f;
    return p;
}

// The closures that the neighbours of a fresh cell (v, w in place) need, one of three
// each: P(w + v) - P(w) as the steps take it, as the FAS right-hand side does, P(w).
__device__ __forceinline__ void close32(const Tail32& t, int l, int q, int part)
{
    const Level<float>& L = t.L[l];
    const C4 w = *t.own(l, W, q);
    if (part == 2) {
        C4 p;
        closure(w.E, w.Fx, w.Fy, L.ic2, p.E, p.Fx, p.Fy);
        p.T = 0.f;
        *t.own(l, E0, q) = p;
        return;
    }
    const C4 v = *t.own(l, V, q);
    if (part == 0) *t.own(l, P0, q) = closure32<false>(L, w, v);
    else *t.own(l, P0 + 1, q) = closure32<true>(L, w, v);
}

// The FAS right-hand side (k_fas_aw32): A(w) and f = [A(w + v) - A(w)] + r.
__device__ __forceinline__ void op_fas(const Tail32& t, int l, int k, int q, int i, int j)
{
    const Level<float>& L = t.L[l];
    const Sig2<float> sg = *t.sig(l, q);
    const C4 w = *t.own(l, W, q), v = *t.own(l, V, q), r = *t.own(l, F, q);
    *t.own(l, AW, q) = base_rows_x(L, sg, w, sums32(t, l, W, E0, true, false, k, q, i, j));
    *t.own(l, F, q) = fas_rhs_x(L, sg, w.T, v, r, sums32(t, l, V, P0 + 1, false, false, k, q, i, j));
}

// One pseudo-time step (the strips' update_cell) from the iterate in array ae with
// closures ap, into buffer `out`.
__device__ __forceinline__ void op_step(const Tail32& t, int l, int ae, int ap, int out, int k, int q,
                                        int i, int j, const Pseudo<float>& ps, unsigned& fails)
{
    const Level<float>& L = t.L[l];
    const Sums32 N = sums32(t, l, ae, ap, false, (t.ring >> l) & 1u, k, q, i, j);
    const C4 u = *t.own(l, ae, q), b = *t.own(l, F, q), w = *t.own(l, W, q), a = *t.own(l, AW, q);
    bool ok;
    const C4 o = pseudo_x(L, *t.sig(l, q), w, a, u, b, N, ps, ok);
    if (!ok) ++fails;
    *t.own(l, E0 + out, q) = o;
    *t.own(l, P0 + out, q) = closure32<false>(L, w, o);
}

// r = f - [A(w + e) - A(w)], into the iterate's other buffer.
__device__ __forceinline__ void op_resid(const Tail32& t, int l, int cur, int k, int q, int i, int j)
{
    const Sums32 N = sums32(t, l, E0 + cur, P0 + cur, false, false, k, q, i, j);
    const C4 u = *t.own(l, E0 + cur, q), b = *t.own(l, F, q);
    *t.own(l, E0 + 1 - cur, q) =
        sub_x(b, rows_x(t.L[l], *t.sig(l, q), t.own(l, W, q)->T, u, N));
}

// One of three arrays (0: v from the iterate, 1: f from the residual, 2: w) of cell
// (i, j) of level l from level l - 1 (k_restrict).  c: the iterate's buffer there, the residual in the other.
__device__ __forceinline__ void op_restrict(const Tail32& t, int l, int c, int q, int i, int j, int part)
{
    const Level<float>& Lf = t.L[l - 1];
    const bool two_d = Lf.dim == 2;
    const int arr = part == 0 ? E0 + c : part == 1 ? E0 + 1 - c : (int)W;
    const int kind = part == 2 ? KIND_STATE : KIND_DIFF;
    const StencilAxis x = stencil_axis(2 * i, Lf.nx, Lf.bc[WALL_W]), y = stencil_axis(2 * j, Lf.ny, Lf.bc[WALL_S]);
    const bool inflow = x.rule == BC_INFLOW || (two_d && y.rule == BC_INFLOW);
    C4 s = { 0, 0, 0, 0 };
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (!two_d && b != 1) continue;
        const float wy = two_d ? (b == 1 ? 0.5f : 0.25f) : 1.f;
        C4 v[3];
        if (!inflow) {
            const int row = two_d ? y.k[b] * Lf.nx : 0;
#pragma unroll
            for (int a = 0; a < 3; ++a) v[a] = *t.at(l - 1, arr, row + x.k[a]);
            if (two_d && b == 0 && y.rule == BC_REFLECT)
#pragma unroll
                for (int a = 0; a < 3; ++a) v[a].Fy = -v[a].Fy;
            if (x.rule == BC_REFLECT) v[0].Fx = -v[0].Fx;
        } else {
            for (int a = 0; a < 3; ++a) {
                const Ghost g = ghost_map(Lf, 2 * i + a - 1, two_d ? 2 * j + b - 1 : 0);
                v[a] = ghost_apply(Lf, *t.at(l - 1, arr, (int)g.k), g, kind);
            }
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float wt = wy * (a == 1 ? 0.5f : 0.25f);
            s = axpy_x(s, wt, v[a]);
        }
    }
    *t.own(l, part == 0 ? (int)V : part == 1 ? (int)F : (int)W, q) = s;
}

// k_prolong onto cell (i, j) of level l; c: the coarse iterate's buffer.
__device__ __forceinline__ void op_prolong(const Tail32& t, int l, int cur, int c, int q, int i, int j,
                                           float theta_c, unsigned& damped)
{
    const Level<float>&L = t.L[l], &Lc = t.L[l + 1];
    const bool two_d = L.dim == 2;
    const int ic = i >> 1, jc = two_d ? j >> 1 : 0, ox = i & 1, oy = two_d ? j & 1 : 0;
    const float wt = pow2_neg<float>(ox + oy);
    // the coarse cells past the high walls under the rules of differences (a cell read
    // with weight zero is not added: sums stay those of k_prolong)
    const bool xo = ic + 1 == Lc.nx, yo = two_d && jc + 1 == Lc.ny;
    const int bx = Lc.bc[WALL_E], by = Lc.bc[WALL_N];
    const int xk = !xo ? ic + 1 : bx == BC_PERIODIC ? 0 : ic, yk = !yo ? jc + 1 : by == BC_PERIODIC ? 0 : jc;
    C4 d[2][2];
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            if (b > oy || a > ox) continue;
            const C4* p = t.at(l + 1, E0, (b ? yk : jc) * Lc.nx + (a ? xk : ic));
            const int per = t.geo[l + 1].per;          // the arrays lie 16 per bytes apart
            const C4 cu = p[c * per], cv = p[(V - E0) * per];
            C4& x = d[b][a];
            x = sub_x(cu, cv);
            if (b && yo && by == BC_REFLECT) x.Fy = -x.Fy;
            if (a && xo && bx == BC_REFLECT) x.Fx = -x.Fx;
            if ((b && yo && by == BC_INFLOW) || (a && xo && bx == BC_INFLOW)) x = C4{ 0, 0, 0, 0 };
        }
    C4 pe = { 0, 0, 0, 0 };
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            if (b > oy || a > ox) continue;
            pe = axpy_x(pe, wt, d[b][a]);
        }
    const C4 w = *t.own(l, W, q);
    bool limited;
    const C4 o = prolong_x(*t.own(l, E0 + cur, q), w, pe, theta_c, L.c, limited);
    if (limited) ++damped;
    *t.own(l, E0 + cur, q) = o;
    *t.own(l, P0 + cur, q) = closure32<false>(L, w, o);
}

// Items are (instance, first tail level), one cluster each (k_tail's loop).
__global__ void __launch_bounds__(kThreads32, 1) k_tail32(const Level<float>* __restrict__ lv, int cap,
                                                          int nlev, WorkList wl,
                                                          Ctl* __restrict__ ctls,
                                                          const unsigned char* __restrict__ prog,
                                                          const int2* __restrict__ progs,
                                                          unsigned ring)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Level<float> Ls[kTailLevels];
    __shared__ Geo32 geo[kTailLevels];
    cg::cluster_group cl = cg::this_cluster();
    const int nb = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int w0 = blockIdx.x / nb, ws = gridDim.x / nb;
    const int nw = *wl.count;
    for (int w = w0; w < nw; w += ws) {
        const int2 it = wl.items[w];
        if (skip(ctls, it.x)) continue;            // the same for the whole cluster
        Ctl* ctl = ctls + it.x;
        const int first = it.y, nl = nlev - first;
        Tail32 t{ Ls, geo, smem, rank, ring >> first, cl };
        const Level<float>* src = lv + (size_t)first * cap + it.x;
        static_assert(sizeof(Level<float>) % 8 == 0 && sizeof(Level<float>) <= 32 * 8, "one word per lane");
        for (int l = threadIdx.x / 32; l < nl; l += kThreads32 / 32) {
            const unsigned long long* s =
                reinterpret_cast<const unsigned long long*>(src + (size_t)l * cap);
            if ((threadIdx.x & 31) < sizeof(Level<float>) / 8)
                reinterpret_cast<unsigned long long*>(&Ls[l])[threadIdx.x & 31] = s[threadIdx.x & 31];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int off = 0;
            for (int l = 0; l < nl; ++l) {
                Geo32 g;
                g.nx = Ls[l].nx;
                g.n = Ls[l].n;
                g.per = tail32_per(g.n, nb);
                g.blocks = (g.n + g.per - 1) / g.per;
                g.off = off;
                g.mx = g.nx > 1 ? (unsigned)((0x100000000ull + g.nx - 1) / g.nx) : 0u;
                g.mper = (unsigned)((0x100000000ull + g.per - 1) / g.per);
                geo[l] = g;
                off += kBytes32 * g.per;
            }
        }
        __syncthreads();
        const Pseudo<float> ps = pseudo_of<float>(ctl);
        const float theta_c = (float)ctl->theta_c;
        unsigned fails = 0, damped = 0;
        for (int l = 0; l < nl; ++l)
            for (int q = threadIdx.x; q < geo[l].per; q += kThreads32) {
                const int k = rank * geo[l].per + q;
                if (k >= geo[l].n) break;
                *t.sig(l, q) = Ls[l].sig[k];
                if (l == 0) {
                    *t.own(0, V, q) = Ls[0].v[k];
                    *t.own(0, W, q) = Ls[0].w[k];
                    *t.own(0, F, q) = Ls[0].r[k];
                    for (int part = 0; part < 3; ++part) close32(t, 0, q, part);
                }
            }
        unsigned curs = 0;                          // bit l: the buffer of level l's iterate
        const int2 pr = progs[first];
        bool was_multi = true;
        for (int p = 0; p <= pr.y; ++p) {
            const int code = p < pr.y ? prog[pr.x + p] : 0;
            const int op = code & 7, l = code >> 3;
            // the levels the operation reads or writes: l and (restriction, prolongation) one
            // more; a single block works while all of them lie in block 0
            const int lo = p == pr.y ? 0 : (op == TAIL_RESTRICT ? l - 1 : l);
            const bool multi = geo[lo].blocks > 1;
            if (multi || was_multi) cl.sync();
            else if (rank == 0) __syncthreads();
            was_multi = multi;
            if (p == pr.y) break;
            const int cur = (curs >> l) & 1;
            const Geo32& g = geo[l];
            const int base = rank * g.per, end = min(g.per, g.n - base);
            const bool two_d = Ls[l].dim == 2;
            if (op == TAIL_RESTRICT) {
                // three threads a cell, an array each; then a closure each
                const int c = (curs >> (l - 1)) & 1;
                for (int x = threadIdx.x; x < 3 * end; x += kThreads32) {
                    const int part = x / end, q = x - part * end, k = base + q;
                    const int j = two_d ? row32(g, k) : 0;
                    op_restrict(t, l, c, q, k - j * g.nx, j, part);
                }
                if (end > 0) __syncthreads();
                for (int x = threadIdx.x; x < 3 * end; x += kThreads32) {
                    const int part = x / end;
                    close32(t, l, x - part * end, part);
                }
                continue;
            }
            for (int q = threadIdx.x; q < end; q += kThreads32) {
                const int k = base + q, j = two_d ? row32(g, k) : 0, i = k - j * g.nx;
                switch (op) {
                case TAIL_FAS: op_fas(t, l, k, q, i, j); break;
                case TAIL_FIRST:
                case TAIL_PSEUDO:
                    op_step(t, l, op == TAIL_FIRST ? (int)V : E0 + cur, op == TAIL_FIRST ? (int)P0 : P0 + cur,
                            op == TAIL_FIRST ? 1 : 1 - cur, k, q, i, j, ps, fails);
                    break;
                case TAIL_RESID: op_resid(t, l, cur, k, q, i, j); break;
                default: op_prolong(t, l, cur, (curs >> (l + 1)) & 1, q, i, j, theta_c, damped); break;
                }
            }
            if (op == TAIL_FIRST) curs |= 1u << l;
            else if (op == TAIL_PSEUDO) curs ^= 1u << l;
        }
        // the result into both buffers of the tail's first level (the other instances of the
        // level decide which one the prolongation reads)
        for (int q = threadIdx.x; q < geo[0].per; q += kThreads32) {
            const int k = rank * geo[0].per + q;
            if (k >= geo[0].n) break;
            const C4 o = *t.own(0, E0 + (curs & 1), q);
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

size_t tail32_smem(int n0, int nb, int dim, int nlev)
{
    size_t s = 0;
    for (int l = 0; l < nlev; ++l) {
        s += (size_t)kBytes32 * tail32_per(n0, nb);
        n0 /= dim == 2 ? 4 : 2;
    }
    return s;
}

cudaError_t tail32_prepare()
{
    const cudaError_t e =
        cudaFuncSetAttribute(k_tail32, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_tail32, cudaFuncAttributeMaxDynamicSharedMemorySize, kTail32Smem);
}

cudaError_t launch_tail32(const Level<float>* lv, int cap, int nlev, WorkList wl, Ctl* ctls,
                          const unsigned char* prog, const int2* progs, unsigned ring, size_t smem,
                          int blocks, cudaStream_t s)
{
    const int most = kTailClusters * kTailBlocks / blocks;
    const int clusters = wl.capacity < most ? (wl.capacity > 0 ? wl.capacity : 1) : most;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * blocks);
    cfg.blockDim = dim3(kThreads32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = blocks;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_tail32, lv, cap, nlev, wl, ctls, prog, progs, ring);
}

}  // namespace m1
