// The FP32 correction-form arithmetic of the coarse levels with every rounding written
// out, one cell at a time.
//
// A coarse level of a mixed instance is walked by the strip kernels (m1_kernels.cu) or
// by the one-launch tail (m1_tail32.cu), as the number of instances beside it decides, and
// a small mixed problem carries last-bit differences into the ninth digit of its result.
// Left to the compiler, fused multiply-adds are chosen kernel by kernel.  Both call these
// functions, so that a level gives the same bits in either whatever the constants and the
// compiler.  Where a choice is stated below it is the one that the strip kernels were
// compiled with when the forms were fixed.
#pragma once
#include "m1_cell.cuh"

namespace m1 {

#define X_MUL __fmul_rn
#define X_ADD __fadd_rn
#define X_SUB(a, b) __fadd_rn((a), -(b))
#define X_FMA __fmaf_rn

// closure_delta.  FAS: as the kernel of the FAS right-hand side sums f0^2 (the y
// term's product fused), else as the sweeps and the residual do (the x term's).
template <bool FAS>
__device__ __forceinline__ void closure_delta_x(float wE, float wFx, float wFy, float eE, float eFx,
                                                float eFy, float ic2, float& dPxx, float& dPxy,
                                                float& dPyy)
{
    const float E1 = X_ADD(wE, eE), iE0 = Fm<float>::rcp(wE), iE1 = Fm<float>::rcp(E1);
    const float px0 = X_MUL(wFx, iE0), py0 = X_MUL(wFy, iE0);
    const float dpx = X_MUL(X_FMA(-px0, eE, eFx), iE1), dpy = X_MUL(X_FMA(-py0, eE, eFy), iE1);
    const float px1 = X_ADD(px0, dpx), py1 = X_ADD(py0, dpy);
    const float f20 = X_MUL(FAS ? X_FMA(py0, py0, X_MUL(px0, px0)) : X_FMA(px0, px0, X_MUL(py0, py0)),
                            ic2);
    const float sx = X_ADD(px0, px1), sy = X_ADD(py0, py1);
    const float df2 = X_MUL(X_FMA(dpx, sx, X_MUL(dpy, sy)), ic2);
    const float f21 = X_ADD(f20, df2);
    const float c0 = f20 < 1.f ? f20 : 1.f, c1 = f21 < 1.f ? f21 : 1.f;
    const float dc = (f20 <= 1.f && f21 <= 1.f) ? df2 : X_SUB(c1, c0);
    const float s0 = Fm<float>::sqrt(X_FMA(-3.f, c0, 4.f)), s1 = Fm<float>::sqrt(X_FMA(-3.f, c1, 4.f));
    const float ds = X_MUL(X_MUL(-3.f, dc), Fm<float>::rcp(X_ADD(s0, s1)));
    const float a1 = X_MUL(X_SUB(s1, 1.f), 1.f / 3.f), da = X_MUL(ds, 1.f / 3.f);
    const float i20 = Fm<float>::rcp(X_ADD(2.f, s0)), i21 = Fm<float>::rcp(X_ADD(2.f, s1));
    const float q0 = X_MUL(3.f, i20), dq = X_MUL(X_MUL(X_MUL(-3.f, ds), i20), i21);
    const float iso = X_FMA(eE, a1, X_MUL(wE, da)), dE = X_MUL(dq, E1);
    const float dEx = X_MUL(dE, px1), dEy = X_MUL(dE, py1), ex = X_MUL(eE, px1), ey = X_MUL(eE, py1);
    dPxx = X_FMA(ic2, X_FMA(q0, X_FMA(ex, px1, X_MUL(X_MUL(wE, dpx), sx)), X_MUL(dEx, px1)), iso);
    dPyy = X_FMA(ic2, X_FMA(q0, X_FMA(ey, py1, X_MUL(X_MUL(wE, dpy), sy)), X_MUL(dEy, py1)), iso);
    dPxy = X_MUL(ic2, X_FMA(q0, X_FMA(ex, py1, X_MUL(wE, X_FMA(px0, dpy, X_MUL(dpx, py1)))),
                            X_MUL(dEx, py1)));
}

// (T + x)^4 - T^4: in the local solve (SOLVE) and in the rows of the operator.
template <bool SOLVE>
__device__ __forceinline__ float quartic_delta_x(float T, float x)
{
    const float t6 = X_MUL(6.f, T), t4 = X_MUL(X_MUL(4.f, T), T), i1 = X_FMA(4.f, T, x);
    const float i2 = SOLVE ? X_FMA(x, i1, X_MUL(t6, T)) : X_FMA(t6, T, X_MUL(x, i1));
    const float i3 = SOLVE ? X_FMA(x, i2, X_MUL(t4, T)) : X_FMA(t4, T, X_MUL(x, i2));
    return X_MUL(x, i3);
}

// local_solve_delta of a pseudo-time step ((w0, w1) = (1, dtau)); dk = diag + kt.
__device__ __forceinline__ Cell4<float> local_solve_delta_x(float dtau, float diag, float ka, float dk,
                                                            float c_v, float a_r, float T, float bE,
                                                            float bFx, float bFy, float bT, bool& ok)
{
    Cell4<float> o;
    const float A = X_FMA(dtau, diag, 1.f), k = X_MUL(dtau, ka), C = X_FMA(dtau, c_v, 1.f);
    const float iF = Fm<float>::rcp(X_FMA(dtau, dk, 1.f));
    o.Fx = X_MUL(bFx, iF);
    o.Fy = X_MUL(bFy, iF);
    ok = true;
    if (k == 0.f) {
        o.T = bT / C;
        o.E = bE / A;
        return o;
    }
    const float iAk = Fm<float>::rcp(X_ADD(A, k));
    const float K = X_MUL(X_MUL(X_MUL(k, A), a_r), iAk), R = X_FMA(X_MUL(k, bE), iAk, bT);
    const float K4 = X_MUL(4.f, K);
    float x = 0.f;
    ok = false;
    for (int it = 0; it < 40; ++it) {
        const float Tx = X_ADD(T, x);
        const float h = X_SUB(X_FMA(C, x, X_MUL(K, quartic_delta_x<true>(T, x))), R);
        const float dh = X_FMA(X_MUL(X_MUL(K4, Tx), Tx), Tx, C);
        const float dx = X_MUL(h, Fm<float>::rcp(dh));
        x = X_SUB(x, dx);
        if (fabsf(dx) <= X_MUL(1e-6f, fabsf(x)) || dx == 0.f) { ok = true; break; }
    }
    o.T = x;
    o.E = X_MUL(X_FMA(X_MUL(k, a_r), quartic_delta_x<true>(T, x), bE), iAk);
    return o;
}

// max_admissible_step; PROLONG: as the prolongation sums |dF|^2 (the y term's product
// fused), else as the pseudo-time step does.
template <bool PROLONG>
__device__ __forceinline__ float max_admissible_step_x(const Cell4<float>& u, const Cell4<float>& d,
                                                       float c)
{
    float tau = INFINITY;
    if (d.E < 0.f) tau = fminf(tau, -u.E / d.E);
    if (d.T < 0.f) tau = fminf(tau, -u.T / d.T);
    const float c2 = X_MUL(c, c), cd = X_MUL(c2, d.E), cu = X_MUL(c2, u.E);
    const float dF2 = PROLONG ? X_FMA(d.Fy, d.Fy, X_MUL(d.Fx, d.Fx)) : X_FMA(d.Fx, d.Fx, X_MUL(d.Fy, d.Fy));
    const float a = X_FMA(-cd, d.E, dF2);
    const float b = X_FMA(-cu, d.E, X_FMA(u.Fx, d.Fx, X_MUL(u.Fy, d.Fy)));
    float c0 = X_FMA(-cu, u.E, X_FMA(u.Fx, u.Fx, X_MUL(u.Fy, u.Fy)));
    c0 = c0 > 0.f ? 0.f : c0;
    const float disc = X_FMA(b, b, -X_MUL(a, c0));
    float t = INFINITY;
    if (a > 0.f) {
        const float sd = sqrtf(disc);
        t = b <= 0.f ? X_ADD(-b, sd) / a : -c0 / X_ADD(b, sd);
    } else if (a < 0.f) {
        if (b > 0.f && disc >= 0.f) t = -c0 / X_ADD(b, sqrtf(disc));
    } else if (b > 0.f) {
        t = -c0 / X_MUL(2.f, b);
    }
    return fminf(tau, t);
}

// admissible_c2 (SLACK as there).
template <bool SLACK>
__device__ __forceinline__ bool admissible_x(const Cell4<float>& s, float c2)
{
    float lim = X_MUL(X_MUL(c2, s.E), s.E);
    if (SLACK) lim = X_MUL(lim, 1.f + Slack<float>::v);
    return s.E > 0.f && s.T > 0.f && X_FMA(s.Fx, s.Fx, X_MUL(s.Fy, s.Fy)) <= lim;
}

__device__ __forceinline__ Cell4<float> add_x(const Cell4<float>& a, const Cell4<float>& b)
{
    return Cell4<float>{ X_ADD(a.E, b.E), X_ADD(a.Fx, b.Fx), X_ADD(a.Fy, b.Fy), X_ADD(a.T, b.T) };
}

// fma by one factor: a + s b.
__device__ __forceinline__ Cell4<float> axpy_x(const Cell4<float>& a, float s, const Cell4<float>& b)
{
    return Cell4<float>{ X_FMA(s, b.E, a.E), X_FMA(s, b.Fx, a.Fx), X_FMA(s, b.Fy, a.Fy),
                         X_FMA(s, b.T, a.T) };
}

__device__ __forceinline__ float limited_step_x(const Cell4<float>& u, const Cell4<float>& f,
                                                float dtau, float theta, float s, float c)
{
    if (admissible_x<false>(axpy_x(u, s, f), X_MUL(c, c))) return dtau;
    return fminf(dtau, X_MUL(theta, max_admissible_step_x<false>(u, f, c)));
}

// The neighbour sums N of Eq. (9): the y pair's term fused onto the x pair's product,
// or (xfused: the strips that stage their rows by cp.async) the other way round.
__device__ __forceinline__ void sums_x(float c, float bx, float by, bool two_d, bool xfused,
                                       const Staged<float>& w, const Staged<float>& e,
                                       const Staged<float>& s, const Staged<float>& n, float& NE, float& NFx, float& NFy)
{
    const float cbx = X_MUL(c, bx), cby = X_MUL(c, by);
    const float xE = X_FMA(c, X_ADD(w.E, e.E), X_SUB(w.Fx, e.Fx));
    const float xF = X_FMA(c, X_SUB(w.Pxx, e.Pxx), X_ADD(w.Fx, e.Fx));
    const float xG = X_FMA(c, X_SUB(w.Pxy, e.Pxy), X_ADD(w.Fy, e.Fy));
    if (!two_d) {
        NE = X_MUL(bx, xE); NFx = X_MUL(cbx, xF); NFy = X_MUL(cbx, xG);
        return;
    }
    const float yE = X_FMA(c, X_ADD(s.E, n.E), X_SUB(s.Fy, n.Fy));
    const float yF = X_FMA(c, X_SUB(s.Pxy, n.Pxy), X_ADD(s.Fx, n.Fx));
    const float yG = X_FMA(c, X_SUB(s.Pyy, n.Pyy), X_ADD(s.Fy, n.Fy));
    if (xfused) {
        NE = X_FMA(bx, xE, X_MUL(by, yE));
        NFx = X_FMA(cbx, xF, X_MUL(cby, yF));
        NFy = X_FMA(cbx, xG, X_MUL(cby, yG));
    } else {
        NE = X_FMA(by, yE, X_MUL(bx, xE));
        NFx = X_FMA(cby, yF, X_MUL(cbx, xF));
        NFy = X_FMA(cby, yG, X_MUL(cbx, xG));
    }
}

// The neighbour sums of a cell.
struct Sums32 {
    float E, Fx, Fy;
};

// One pseudo-time step of a cell (update_cell's correction form): its base w, A(w), iterate
// e and right-hand side b.
__device__ __forceinline__ Cell4<float> pseudo_x(const Level<float>& L, const Sig2<float>& sg,
                                                 const Cell4<float>& w, const Cell4<float>& aw,
                                                 const Cell4<float>& e, const Cell4<float>& b,
                                                 const Sums32& N, const Pseudo<float>& ps, bool& ok)
{
    const float ka = X_MUL(L.cdt, sg.sa), dk = X_ADD(L.diag, X_MUL(L.cdt, X_ADD(sg.sa, sg.ss)));
    const float tau = limited_step_x(add_x(w, e), add_x(aw, b), ps.dtau, ps.theta, ps.s, L.c);
    const float lim = X_SUB(tau, ps.dtau);
    const Cell4<float> rhs = axpy_x(axpy_x(e, tau, b), lim, aw);
    return local_solve_delta_x(ps.dtau, L.diag, ka, dk, L.c_v, L.a_r, w.T, X_FMA(ps.dtau, N.E, rhs.E),
                               X_FMA(ps.dtau, N.Fx, rhs.Fx), X_FMA(ps.dtau, N.Fy, rhs.Fy), rhs.T, ok);
}

// A(w + e) - A(w) of a cell of base temperature T.
__device__ __forceinline__ Cell4<float> rows_x(const Level<float>& L, const Sig2<float>& sg, float T,
                                               const Cell4<float>& e, const Sums32& N)
{
    const float ka = X_MUL(L.cdt, sg.sa), dk = X_FMA(L.cdt, X_ADD(sg.sa, sg.ss), L.diag);
    const float se = X_MUL(ka, X_FMA(-L.a_r, quartic_delta_x<false>(T, e.T), e.E));
    return Cell4<float>{ X_SUB(X_FMA(L.diag, e.E, se), N.E), X_FMA(dk, e.Fx, -N.Fx),
                         X_FMA(dk, e.Fy, -N.Fy), X_FMA(L.c_v, e.T, -se) };
}

__device__ __forceinline__ Cell4<float> sub_x(const Cell4<float>& a, const Cell4<float>& b)
{
    return Cell4<float>{ X_SUB(a.E, b.E), X_SUB(a.Fx, b.Fx), X_SUB(a.Fy, b.Fy), X_SUB(a.T, b.T) };
}

// The right-hand side of a fresh visit: A(w), from the sums of w, and
// f = [A(w + v) - A(w)] + r, from those of v.
__device__ __forceinline__ Cell4<float> base_rows_x(const Level<float>& L, const Sig2<float>& sg,
                                                    const Cell4<float>& w, const Sums32& N)
{
    const float ka = X_MUL(L.cdt, sg.sa), dk = X_ADD(L.diag, X_MUL(L.cdt, X_ADD(sg.sa, sg.ss)));
    const float T2 = X_MUL(w.T, w.T), sw = X_MUL(ka, X_FMA(-X_MUL(L.a_r, T2), T2, w.E));
    return Cell4<float>{ X_SUB(X_FMA(L.diag, w.E, sw), N.E), X_FMA(dk, w.Fx, -N.Fx),
                         X_FMA(dk, w.Fy, -N.Fy), X_FMA(L.c_v, w.T, -sw) };
}
__device__ __forceinline__ Cell4<float> fas_rhs_x(const Level<float>& L, const Sig2<float>& sg, float T,
                                                  const Cell4<float>& v, const Cell4<float>& r,
                                                  const Sums32& N)
{
    const float ka = X_MUL(L.cdt, sg.sa), dk = X_ADD(L.diag, X_MUL(L.cdt, X_ADD(sg.sa, sg.ss)));
    const float sd = X_MUL(ka, X_FMA(-L.a_r, quartic_delta_x<false>(T, v.T), v.E));
    return add_x(Cell4<float>{ X_SUB(X_FMA(L.diag, v.E, sd), N.E), X_FMA(dk, v.Fx, -N.Fx),
                               X_FMA(dk, v.Fy, -N.Fy), X_FMA(L.c_v, v.T, -sd) }, r);
}

// The correction e of a fine cell of base w with the prolongated correction pe added,
// damped (Eq. (34)) where the target is not admissible.
__device__ __forceinline__ Cell4<float> prolong_x(const Cell4<float>& e, const Cell4<float>& w,
                                                  const Cell4<float>& pe, float theta_c, float c,
                                                  bool& damped)
{
    const Cell4<float> u = add_x(e, w);
    damped = !admissible_x<true>(add_x(u, pe), X_MUL(c, c));
    const float th = damped ? X_MUL(theta_c, fminf(1.f, max_admissible_step_x<true>(u, pe, c))) : 1.f;
    return axpy_x(e, th, pe);
}

}  // namespace m1
