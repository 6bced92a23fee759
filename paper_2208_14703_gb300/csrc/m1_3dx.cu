// The 3D passes in fixed point (m1_3fx.cuh): one pass a sweep, each forming its
// result's blocks for the next one.
//
// What bounds them: instruction issue and, on grids over L2, the planes' traffic
// (a Jacobi sweep reads about 96 bytes of blocks, 40 of b, 32 of coefficients and
// writes 136 a cell).  The FP64 form (m1_3d.cu), a closure pass and an operator
// pass, is bound by the FP64 pipe at about 150 operations a cell; it stays for
// grids whose blocks do not fit the device and for cells no block can hold.
#include "m1_3fx.cuh"

namespace m1 {
namespace {

constexpr int kThreadsX3 = 128;
constexpr int kMaxBlocksX3 = 152 * 8 * 2;

__device__ __forceinline__ bool skipx3(const Ctl* ctl) { return ctl && ctl->done; }

// The whole neighbour sums of a cell in FP64 (some block of its stencil is irregular).
__device__ __noinline__ void general_sums3(const G3& g, const EF* __restrict__ u, int i, int j, int k,
                                           double N[4])
{
    N[0] = N[1] = N[2] = N[3] = 0.0;
    for (int d = 0; d < 3; ++d)
        for (int side = -1; side <= 1; side += 2) {
            int p[3] = { i, j, k };
            p[d] += side;
            EF nb;
            int rule = -1;                       // fetch3's rules for a state
            if (p[d] < 0 || p[d] >= g.n[d]) {
                const int bc = g.bc[2 * d + (side < 0 ? 0 : 1)];
                if (bc == BC_PERIODIC) p[d] = p[d] < 0 ? p[d] + g.n[d] : p[d] - g.n[d];
                else if (bc != BC_INFLOW) p[d] = p[d] < 0 ? 0 : g.n[d] - 1;
                if (bc != BC_PERIODIC) rule = bc;
            }
            if (rule == BC_INFLOW) inflow_at(g, d, side < 0 ? 0 : 1, p, nb);
            else nb = u[at3(g, p[0], p[1], p[2])];
            if (rule == BC_REFLECT) nb.F[d] = -nb.F[d];
            const P6 pn = closure3(nb, g.ic2);
            const double sg = side < 0 ? 1.0 : -1.0, bd = g.beta[d];
            N[0] += bd * (g.c * nb.E + sg * nb.F[d]);
            for (int a = 0; a < 3; ++a)
                N[1 + a] += g.c * bd * (nb.F[a] + sg * g.c * P_at(pn, d, a));
        }
}

__device__ __forceinline__ double limited_step3(const EF& u, double T, const EF& f, double fT,
                                                double dtau, double theta, double c,
                                                const ConeScale& cone)
{
    FluxSum F(cone);
#pragma unroll
    for (int a = 0; a < 3; ++a) F.add(u.F[a], f.F[a]);
    if (admissible_sure(u.E, T, f.E, fT, F) > 0) return dtau;
    const double cd = c * c * f.E, cu = c * c * u.E;
    double a = -cd * f.E, b = -cu * f.E, c0 = -cu * u.E;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        a = fma(f.F[m], f.F[m], a);
        b = fma(u.F[m], f.F[m], b);
        c0 = fma(u.F[m], u.F[m], c0);
    }
    return fmin(dtau, theta * fmin(fmin(plane_step(u.E, f.E), plane_step(T, fT)), cone_step(a, b, c0)));
}

__device__ __forceinline__ Coef coef3(const G3& g, double w0, double w1, const Sig2<double>& s)
{
    return make_coef(w0, w1, g.diag, g.cdt * s.sa, g.cdt * (s.sa + s.ss), g.a_r);
}

// local_solve64 with three flux components.
__device__ __forceinline__ void solvex3(const Coef& q, double A, double C, double a_r, double bE,
                                        const double bF[3], double bT, EF& o, double& oT, bool& ok)
{
    const Cell4<double> r = local_solve64(q, A, C, a_r, bE, bF[0], bF[1], bT, ok);
    o.E = r.E;
    o.F[0] = r.Fx;
    o.F[1] = r.Fy;
    o.F[2] = bF[2] * q.iF;
    oT = r.T;
}

// A cell of a state: EF and T arrays, or (PLANAR) the five planes of a caller's array.
template <bool PLANAR>
__device__ __forceinline__ EF load3(const EF* __restrict__ x, size_t n, size_t q)
{
    if (!PLANAR) return x[q];
    const double* p = reinterpret_cast<const double*>(x);
    return EF{ p[q], { p[n + q], p[2 * n + q], p[3 * n + q] } };
}

template <bool PLANAR>
__device__ __forceinline__ void store3(EF* __restrict__ x, size_t n, size_t q, const EF& v)
{
    if (!PLANAR) {
        x[q] = v;
        return;
    }
    double* p = reinterpret_cast<double*>(x);
    p[q] = v.E;
    p[n + q] = v.F[0];
    p[2 * n + q] = v.F[1];
    p[3 * n + q] = v.F[2];
}

template <bool PLANAR>
__device__ __forceinline__ Sig2<double> opacity3(const Sig2<double>* __restrict__ s, size_t n, size_t q)
{
    if (!PLANAR) return s[q];
    const double* p = reinterpret_cast<const double*>(s);
    return Sig2<double>{ p[q], p[n + q] };
}

// PLANAR (m1_op_level3): the states are a caller's planes, of which intermediate
// sweeps write none (out null: the blocks alone), the coefficients are formed in
// place (FP64 operations the pass has room for, against a pass over the opacities
// and 32 bytes a cell), and a cell with an irregular stencil sets *irregular (the
// caller then takes the FP64 form).
// Six blocks per SM: cycles of 64^3, 128^3 and 192^3 take 0.550, 2.64 and 8.12 ms (5 blocks
// 0.535, 2.81 and 8.82; 7 blocks 0.552, 2.77 and 8.68), four PLANAR sweeps of 192^3 4.27 ms
// (5 blocks 4.61, 7 blocks 4.49).
template <int MODE, bool PLANAR = false>
__global__ void __launch_bounds__(kThreadsX3, 6) k_opx3(G3 g, const EF* __restrict__ u,
                                                     const double* __restrict__ T, Blocks3 B,
                                                     Coef* __restrict__ Q,
                                                     const Sig2<double>* __restrict__ sig,
                                                     const EF* __restrict__ b,
                                                     const double* __restrict__ bT,
                                                     EF* __restrict__ f, double* __restrict__ fT,
                                                     EF* __restrict__ out, double* __restrict__ outT,
                                                     Blocks3 Bo, size_t n, Ctl* __restrict__ ctl,
                                                     double* __restrict__ part,
                                                     int* __restrict__ irregular)
{
    constexpr bool STEP = MODE == OPX3_FIRST || MODE == OPX3_PSEUDO;
    constexpr bool JAC = MODE == OPX3_JACOBI || MODE == OPX3_JACOBI_NORM;
    constexpr bool LOCAL = MODE != OPX3_JACOBI && MODE != OPX3_PSEUDO;   // forms D(u)
    if (skipx3(ctl)) return;
    double dtau = 0.0, theta = 0.0;
    if (STEP) { dtau = ctl->dtau; theta = ctl->theta_ex; }
    const ConeScale cone = STEP ? cone_scale(dtau / theta, g.ic) : ConeScale{};
    const double A = STEP ? fma(dtau, g.diag, 1.0) : g.diag, C = STEP ? fma(dtau, g.c_v, 1.0) : g.c_v;
    double nrm = 0.0;
    unsigned int fails = 0;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x) {
        const unsigned row = (unsigned)q / (unsigned)g.n[0];
        const int p[3] = { (int)((unsigned)q - row * (unsigned)g.n[0]), (int)(row % (unsigned)g.n[1]),
                           (int)(row / (unsigned)g.n[1]) };
        const EF bb = MODE == OPX3_APPLY ? EF{} : load3<PLANAR>(b, n, q);
        const double bbT = MODE == OPX3_APPLY ? 0.0 : bT[q];
        double N[4], fE = g.cb, fF = g.cbF;
        if (!sums3(g, B, n, (unsigned)q, p, N)) {
            if (PLANAR) {
                *irregular = 1;
                continue;
            }
            general_sums3(g, u, p[0], p[1], p[2], N);
            fE = fF = 1.0;
        }
        EF uc{};
        double Tc = 0.0;
        if (!(MODE == OPX3_JACOBI)) { uc = load3<PLANAR>(u, n, q); Tc = T[q]; }
        EF a{};
        double aT = 0.0;
        Sig2<double> sg{};
        if (LOCAL) {
            sg = opacity3<PLANAR>(sig, n, q);
            const double ka = g.cdt * sg.sa, dF = g.diag + g.cdt * (sg.sa + sg.ss);
            const double T2 = Tc * Tc, src = ka * fma(-g.a_r, T2 * T2, uc.E);
            a.E = fma(-fE, N[0], fma(g.diag, uc.E, src));
#pragma unroll
            for (int m = 0; m < 3; ++m) a.F[m] = fma(-fF, N[1 + m], dF * uc.F[m]);
            aT = fma(g.c_v, Tc, -src);
        }
        if (MODE == OPX3_APPLY) {
            store3<PLANAR>(out, n, q, a);
            outT[q] = aT;
            continue;
        }
        if (MODE == OPX3_RESID || MODE == OPX3_JACOBI_NORM) {
            EF r;
            r.E = bb.E - a.E;
#pragma unroll
            for (int m = 0; m < 3; ++m) r.F[m] = bb.F[m] - a.F[m];
            const double rT = bbT - aT;
            nrm += fma(fma(r.F[2], r.F[2], fma(r.F[1], r.F[1], r.F[0] * r.F[0])), g.ic2,
                       fma(r.E, r.E, rT * rT));
            if (MODE == OPX3_RESID) {
                store3<PLANAR>(out, n, q, r);
                outT[q] = rT;
                continue;
            }
        }
        bool ok;
        EF o;
        double oT, rhs[3];
        if (JAC) {
#pragma unroll
            for (int m = 0; m < 3; ++m) rhs[m] = fma(fF, N[1 + m], bb.F[m]);
            solvex3(PLANAR ? coef3(g, 0.0, 1.0, opacity3<PLANAR>(sig, n, q)) : Q[q], A, C, g.a_r, fma(fE, N[0], bb.E), rhs, bbT, o, oT, ok);
        } else {
            EF ff = bb;
            double ffT = bbT;
            Coef co;
            if (MODE == OPX3_FIRST) {
                ff.E += a.E;
#pragma unroll
                for (int m = 0; m < 3; ++m) ff.F[m] += a.F[m];
                ffT += aT;
                f[q] = ff;
                fT[q] = ffT;
                co = coef3(g, 1.0, dtau, sg);
                Q[q] = co;
            } else {
                co = Q[q];
            }
            const double tau = limited_step3(uc, Tc, ff, ffT, dtau, theta, g.c, cone);
#pragma unroll
            for (int m = 0; m < 3; ++m)
                rhs[m] = fma(dtau * fF, N[1 + m], fma(tau, ff.F[m], uc.F[m]));
            solvex3(co, A, C, g.a_r, fma(dtau * fE, N[0], fma(tau, ff.E, uc.E)), rhs,
                    fma(tau, ffT, Tc), o, oT, ok);
        }
        if (!ok) ++fails;
        if (!PLANAR || out) {
            store3<PLANAR>(out, n, q, o);
            outT[q] = oT;
        }
        if (Bo.m) put_block3(g, o, Bo, n, q);
    }
    if (fails && ctl) atomicAdd(&ctl->newton_fail, fails);
    if ((MODE == OPX3_RESID || MODE == OPX3_JACOBI_NORM) && part) {
        __shared__ double red[kThreadsX3];
        red[threadIdx.x] = nrm;
        __syncthreads();
        for (int w = blockDim.x / 2; w > 0; w >>= 1) {
            if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
            __syncthreads();
        }
        if (threadIdx.x == 0) part[blockIdx.x] = red[0] * g.vol;
    }
}

template <bool PLANAR>
__global__ void __launch_bounds__(kThreadsX3) k_blockx3(G3 g, const EF* __restrict__ u, Blocks3 B,
                                                        size_t n, const Ctl* __restrict__ ctl)
{
    if (skipx3(ctl)) return;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x)
        put_block3(g, load3<PLANAR>(u, n, q), B, n, q);
}

__global__ void __launch_bounds__(kThreadsX3) k_coefx3(G3 g, const Sig2<double>* __restrict__ sig,
                                                       Coef* __restrict__ Q, size_t n)
{
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n;
         q += (size_t)gridDim.x * blockDim.x)
        Q[q] = coef3(g, 0.0, 1.0, sig[q]);
}

// Full weighting, one thread per coarse cell and field: 32 coarse cells a block, ten
// warps (E, F, T of the iterate, then of the residual).  A thread's 27 FP64
// multiply-adds are its latency (a thread per cell took ten times as long on the
// small levels); the first warp then forms the blocks of the restricted iterate.
__global__ void __launch_bounds__(320) k_restrictx3(G3 gf, G3 gc, const EF* __restrict__ u,
                                                    const double* __restrict__ uT,
                                                    const EF* __restrict__ r,
                                                    const double* __restrict__ rT,
                                                    EF* __restrict__ vc, double* __restrict__ vcT,
                                                    EF* __restrict__ rc, double* __restrict__ rcT,
                                                    Blocks3 Bo, const Ctl* __restrict__ ctl)
{
    __shared__ double val[4][32];
    if (skipx3(ctl)) return;
    const size_t nc = (size_t)gc.n[0] * gc.n[1] * gc.n[2];
    const int lane = threadIdx.x & 31, field = threadIdx.x >> 5, fl = field % 5;
    const bool state = field < 5;
    const EF* __restrict__ x = state ? u : r;
    const double* __restrict__ xT = state ? uT : rT;
    for (size_t base = (size_t)blockIdx.x * 32; base < nc; base += (size_t)gridDim.x * 32) {
        const size_t q = base + lane;
        if (q < nc) {
            const unsigned row = (unsigned)q / (unsigned)gc.n[0];
            const int ic = (int)((unsigned)q - row * (unsigned)gc.n[0]);
            const int jc = (int)(row % (unsigned)gc.n[1]), kc = (int)(row / (unsigned)gc.n[1]);
            const bool inside = ic > 0 && jc > 0 && kc > 0 && 2 * ic + 1 < gf.n[0] &&
                                2 * jc + 1 < gf.n[1] && 2 * kc + 1 < gf.n[2];
            double acc = 0.0;
            for (int cz = -1; cz <= 1; ++cz)
                for (int by = -1; by <= 1; ++by) {
#pragma unroll
                    for (int ax = -1; ax <= 1; ++ax) {
                        // weights 2^-(3 .. 6): 1/2 at the centre of an axis, 1/4 beside it
                        const double wt = __longlong_as_double(
                            (long long)(1023 - 3 - (cz != 0) - (by != 0) - (ax != 0)) << 52);
                        double s;
                        if (inside) {
                            const size_t k = at3(gf, 2 * ic + ax, 2 * jc + by, 2 * kc + cz);
                            s = fl == 4 ? xT[k] : reinterpret_cast<const double*>(x + k)[fl];
                        } else {
                            EF e;
                            double t;
                            fetch3(gf, x, xT, 2 * ic + ax, 2 * jc + by, 2 * kc + cz,
                                   state ? K3_STATE : K3_DIFF, e, t);
                            s = fl == 0 ? e.E : fl == 4 ? t : e.F[fl - 1];
                        }
                        acc = fma(wt, s, acc);
                    }
                }
            if (fl == 4) (state ? vcT : rcT)[q] = acc;
            else reinterpret_cast<double*>((state ? vc : rc) + q)[fl] = acc;
            if (state && fl < 4) val[fl][lane] = acc;
        }
        __syncthreads();
        if (field == 0 && q < nc) {
            const EF e = { val[0][lane], { val[1][lane], val[2][lane], val[3][lane] } };
            put_block3(gc, e, Bo, nc, q);
        }
        __syncthreads();
    }
}

// Prolongation with damping (k_prolong3's rules), a warp per 31 coarse columns of one
// fine (y, z) row: a lane sums the coarse differences of its column (1, 2 or 4 of
// them), takes its east neighbour's sum by a shuffle, and corrects the two fine cells
// 2 ic (the sum) and 2 ic + 1 (both sums); the weights are powers of two.
__global__ void __launch_bounds__(kThreadsX3) k_prolongx3(G3 gc, G3 gf, const EF* __restrict__ uc,
                                                          const double* __restrict__ ucT,
                                                          const EF* __restrict__ vc,
                                                          const double* __restrict__ vcT,
                                                          EF* __restrict__ uf,
                                                          double* __restrict__ ufT, Blocks3 Bo,
                                                          Ctl* __restrict__ ctl)
{
    if (skipx3(ctl)) return;
    const double theta = ctl->theta_c, c = gf.c;
    const ConeScale cone = cone_scale(1.0, gf.ic);
    const size_t nf = (size_t)gf.n[0] * gf.n[1] * gf.n[2];
    const int lane = threadIdx.x & 31;
    const unsigned chunks = (unsigned)(gc.n[0] + 30) / 31u;
    const size_t items = (size_t)chunks * gf.n[1] * gf.n[2];
    unsigned int damped = 0;
    for (size_t it = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) / 32; it < items;
         it += (size_t)gridDim.x * blockDim.x / 32) {
        const unsigned row = (unsigned)it / chunks;
        const int ic = (int)((unsigned)it - row * chunks) * 31 + lane;
        const int j = (int)(row % (unsigned)gf.n[1]), k = (int)(row / (unsigned)gf.n[1]);
        const int jc = j >> 1, kc = k >> 1, oy = j & 1, oz = k & 1;
        double S[5] = { 0.0, 0.0, 0.0, 0.0, 0.0 };
        if (ic <= gc.n[0]) {
            const bool inside = ic < gc.n[0] && jc + oy < gc.n[1] && kc + oz < gc.n[2];
            for (int cz = 0; cz <= oz; ++cz)
                for (int by = 0; by <= oy; ++by) {
                    EF a, b;
                    double aT, bT;
                    if (inside) {
                        const size_t q = at3(gc, ic, jc + by, kc + cz);
                        a = uc[q]; b = vc[q]; aT = ucT[q]; bT = vcT[q];
                    } else {
                        fetch3(gc, uc, ucT, ic, jc + by, kc + cz, K3_DIFF, a, aT);
                        fetch3(gc, vc, vcT, ic, jc + by, kc + cz, K3_DIFF, b, bT);
                    }
                    S[0] += a.E - b.E;
#pragma unroll
                    for (int m = 0; m < 3; ++m) S[1 + m] += a.F[m] - b.F[m];
                    S[4] += aT - bT;
                }
        }
        double E[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) E[m] = S[m] + __shfl_down_sync(0xffffffffu, S[m], 1);
        if (lane == 31 || ic >= gc.n[0]) continue;
#pragma unroll
        for (int ox = 0; ox < 2; ++ox) {
            const double wt = __longlong_as_double((long long)(1023 - ox - oy - oz) << 52);
            const double* __restrict__ pe = ox ? E : S;
            const size_t q = at3(gf, 2 * ic + ox, j, k);
            const EF u = uf[q];
            const double uT = ufT[q];
            EF t;
            t.E = fma(wt, pe[0], u.E);
#pragma unroll
            for (int m = 0; m < 3; ++m) t.F[m] = fma(wt, pe[1 + m], u.F[m]);
            double tT = fma(wt, pe[4], uT);
            FluxSum F(cone);
#pragma unroll
            for (int m = 0; m < 3; ++m) F.add(t.F[m], 0.0);
            const int sure = admissible_sure(t.E, tT, 0.0, 0.0, F);
            if (sure < 0 || (sure == 0 && !admissible3(t, tT, c))) {
                EF d;
                d.E = wt * pe[0];
                for (int m = 0; m < 3; ++m) d.F[m] = wt * pe[1 + m];
                const double dT = wt * pe[4];
                const double th = theta * fmin(1.0, max_step3(u, uT, d, dT, c));
                t.E = u.E + th * d.E;
                for (int m = 0; m < 3; ++m) t.F[m] = u.F[m] + th * d.F[m];
                tT = uT + th * dT;
                ++damped;
            }
            uf[q] = t;
            ufT[q] = tT;
            put_block3(gf, t, Bo, nf, q);
        }
    }
    if (damped) atomicAdd(&ctl->damped, damped);
}

int gridx3(size_t items, size_t per)
{
    const size_t b = (items + per - 1) / per;
    return (int)(b < (size_t)kMaxBlocksX3 ? (b > 0 ? b : 1) : kMaxBlocksX3);
}

}  // namespace

int blocksx3(size_t n) { return gridx3(n, kThreadsX3); }

void launchx3_block(const G3& g, const EF* u, const Blocks3& B, size_t n, const Ctl* ctl,
                    cudaStream_t s)
{
    k_blockx3<false><<<blocksx3(n), kThreadsX3, 0, s>>>(g, u, B, n, ctl);
}

void launchx3_coef(const G3& g, const Sig2<double>* sig, Coef* Q, size_t n, cudaStream_t s)
{
    k_coefx3<<<blocksx3(n), kThreadsX3, 0, s>>>(g, sig, Q, n);
}

void launchx3_op(int mode, const G3& g, const EF* u, const double* uT, const Blocks3& B, Coef* Q,
                 const Sig2<double>* sig, const EF* b, const double* bT, EF* f, double* fT, EF* out,
                 double* outT, const Blocks3& Bo, size_t n, Ctl* ctl, double* part, cudaStream_t s)
{
    const int nb = blocksx3(n);
    auto go = [&](auto* k) {
        k<<<nb, kThreadsX3, 0, s>>>(g, u, uT, B, Q, sig, b, bT, f, fT, out, outT, Bo, n, ctl, part,
                                    nullptr);
    };
    switch (mode) {
    case OPX3_APPLY: go(k_opx3<OPX3_APPLY>); break;
    case OPX3_RESID: go(k_opx3<OPX3_RESID>); break;
    case OPX3_JACOBI: go(k_opx3<OPX3_JACOBI>); break;
    case OPX3_JACOBI_NORM: go(k_opx3<OPX3_JACOBI_NORM>); break;
    case OPX3_FIRST: go(k_opx3<OPX3_FIRST>); break;
    default: go(k_opx3<OPX3_PSEUDO>); break;
    }
}

void launchx3_planar(int mode, const G3& g, const double* u, const Blocks3& B, const double* sig,
                     const double* b, double* out, const Blocks3& Bo, size_t n, int* irregular,
                     cudaStream_t s)
{
    const int nb = blocksx3(n);
    auto go = [&](auto* k) {
        k<<<nb, kThreadsX3, 0, s>>>(g, reinterpret_cast<const EF*>(u), u + 4 * n, B, nullptr,
                                    reinterpret_cast<const Sig2<double>*>(sig),
                                    reinterpret_cast<const EF*>(b), b ? b + 4 * n : nullptr, nullptr,
                                    nullptr, reinterpret_cast<EF*>(out), out ? out + 4 * n : nullptr,
                                    Bo, n, nullptr, nullptr, irregular);
    };
    if (mode == OPX3_APPLY) go(k_opx3<OPX3_APPLY, true>);
    else if (mode == OPX3_RESID) go(k_opx3<OPX3_RESID, true>);
    else go(k_opx3<OPX3_JACOBI, true>);
}

void launchx3_block_planar(const G3& g, const double* u, const Blocks3& B, size_t n, cudaStream_t s)
{
    k_blockx3<true><<<blocksx3(n), kThreadsX3, 0, s>>>(g, reinterpret_cast<const EF*>(u), B, n, nullptr);
}

void launchx3_restrict(const G3& gf, const G3& gc, const EF* u, const double* uT, const EF* r,
                       const double* rT, EF* vc, double* vcT, EF* rc, double* rcT, const Blocks3& Bo,
                       const Ctl* ctl, cudaStream_t s)
{
    const size_t nc = (size_t)gc.n[0] * gc.n[1] * gc.n[2];
    k_restrictx3<<<gridx3(nc, 32), 320, 0, s>>>(gf, gc, u, uT, r, rT, vc, vcT, rc, rcT, Bo, ctl);
}

void launchx3_prolong(const G3& gc, const G3& gf, const EF* uc, const double* ucT, const EF* vc,
                      const double* vcT, EF* uf, double* ufT, const Blocks3& Bo, Ctl* ctl,
                      cudaStream_t s)
{
    const size_t items = (size_t)((gc.n[0] + 30) / 31) * gf.n[1] * gf.n[2];
    k_prolongx3<<<gridx3(items, kThreadsX3 / 32), kThreadsX3, 0, s>>>(gc, gf, uc, ucT, vc, vcT, uf,
                                                                     ufT, Bo, ctl);
}

}  // namespace m1
