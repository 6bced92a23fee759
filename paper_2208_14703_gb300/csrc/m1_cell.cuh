// Per-cell pieces shared by the stencil kernels (m1_kernels.cu, m1_tail.cu): the
// staged neighbour, its sums, the limited explicit pseudo-time step.
#pragma once
#include "m1_device.cuh"

namespace m1 {

// The explicit pseudo-time step length min(dtau, theta tau*) of Algorithm 3
// (tau* = the largest admissible step from u along f).  The admissible set is
// convex, so when u + (dtau / theta) f is admissible tau* >= dtau / theta and
// the step is dtau: the divisions and the square root of tau* are needed only
// in cells where the bound may bind.  s = dtau / theta is passed in (once per
// strip).
template <typename R>
__device__ __forceinline__ R limited_step(const Cell4<R>& u, const Cell4<R>& f, R dtau, R theta,
                                          R s, R c)
{
    const Cell4<R> p = { u.E + s * f.E, u.Fx + s * f.Fx, u.Fy + s * f.Fy, u.T + s * f.T };
    if (admissible_c2<R, false>(p, c * c)) return dtau;
    return fmin(dtau, theta * max_admissible_step(u, f, c));
}

__device__ __forceinline__ bool skip(const Ctl* ctls, int inst)
{
    return ctls && (ctls[inst].done || !ctls[inst].active);
}

// 2^-k (0 <= k <= 4) built from its exponent: the transfer weights are products
// of 1/2 and 1/4, exact either way, and this keeps them off the FP64 pipe.
template <typename R>
__device__ __forceinline__ R pow2_neg(int k)
{
    if constexpr (sizeof(R) == 8) return __longlong_as_double((long long)(1023 - k) << 52);
    else return __int_as_float((127 - k) << 23);
}

// One cell of a warp strip as its neighbours need it: the state (or, in the
// correction form, the correction e) and its closure P (or P(w + e) - P(w)),
// plus the temperature the cell's own update needs (u.T; correction form: the
// base w.T).
template <typename R>
struct Staged {
    R E, Fx, Fy, Pxx, Pxy, Pyy, T;
};

// The pseudo-time constants of a sweep, read once per strip: dtau_im, theta_ex
// and dtau_im / theta_ex.
template <typename R>
struct Pseudo {
    R dtau, theta, s;
};

template <typename R>
__device__ __forceinline__ Pseudo<R> pseudo_of(const Ctl* ctl)
{
    const double dtau = ctl->dtau, theta = ctl->theta_ex;
    return Pseudo<R>{ (R)dtau, (R)theta, (R)(dtau / theta) };
}

// Neighbour operators L and R of Eq. (9) of a strip cell from its staged west /
// east (shuffled) and south / north rows.
template <typename R>
__device__ __forceinline__ void strip_neighbours(const Level<R>& L, const Staged<R>& wv,
                                                 const Staged<R>& ev, const Staged<R>& prev,
                                                 const Staged<R>& next, bool two_d, R& NE,
                                                 R& NFx, R& NFy)
{
    const R c = L.c, bx = L.bx, by = L.by;
    NE = bx * (c * (wv.E + ev.E) + (wv.Fx - ev.Fx));
    NFx = c * bx * ((wv.Fx + ev.Fx) + c * (wv.Pxx - ev.Pxx));
    NFy = c * bx * ((wv.Fy + ev.Fy) + c * (wv.Pxy - ev.Pxy));
    if (two_d) {
        NE += by * (c * (prev.E + next.E) + (prev.Fy - next.Fy));
        NFx += c * by * ((prev.Fx + next.Fx) + c * (prev.Pxy - next.Pxy));
        NFy += c * by * ((prev.Fy + next.Fy) + c * (prev.Pyy - next.Pyy));
    }
}

// The rows or columns c - 1, c, c + 1 (c even) of an axis of n cells under its low
// wall's rule: indices, and the rule that c - 1 falls under (-1: none, or periodic).
// n is even where this is asked (a level that is restricted), so c + 1 < n.
struct StencilAxis {
    int k[3], rule;
};
__device__ __forceinline__ StencilAxis stencil_axis(int c, int n, int bc)
{
    StencilAxis a = { { c - 1, c, c + 1 }, -1 };
    if (c == 0) {
        a.k[0] = bc == BC_PERIODIC ? n - 1 : 0;
        if (bc != BC_PERIODIC) a.rule = bc;
    }
    return a;
}

}  // namespace m1
