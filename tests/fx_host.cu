// Host entries to the kernels' arithmetic that is host code too (m1_fx.cuh,
// m1_strip64.cuh), for tests that need no GPU (tests/fx_host.py compiles this file).
#include "m1_strip64.cuh"
#include "m1_tail.h"

using namespace m1;

// The FP32 answer to whether u + s f is admissible: n cells [E, Fx, Fy, T] each.
extern "C" void host_admissible_sure(int n, const double* u, const double* f, double s, double c,
                                     int* out)
{
    const ConeScale q = cone_scale(s, 1.0 / c);
    for (int k = 0; k < n; ++k) {
        const double *a = u + 4 * k, *b = f + 4 * k;
        FluxSum F(q);
        F.add(a[1], b[1]);
        F.add(a[2], b[2]);
        out[k] = admissible_sure(a[0], a[3], b[0], b[3], F);
    }
}

extern "C" void host_product(int n, const long long* a, long long b, long long* out)
{
    for (int k = 0; k < n; ++k) out[k] = fx_product(a[k], split62(b));
}

// The neighbour sums of n cells from their four neighbours (west, east, south, north; two
// in 1D), [E, Fx, Fy] each, F over c: out N_E / cb, N_Fx / cbF, N_Fy / cbF; 0 where a
// neighbour is not regular.
extern "C" int host_sums(int n, int dim, const double* cells, double* out)
{
    int regular = 0;
    for (int k = 0; k < n; ++k) {
        FxCell c[4];
        bool ok = true;
        for (int w = 0; w < 2 * dim; ++w) {
            const double* u = cells + (k * 4 + w) * 3;
            ok = fx_stage(u[0], u[1], u[2], c[w]) && ok;
        }
        if (!ok) continue;
        ++regular;
        FxFlux f[4];
        for (int q = 0; q < 2 * dim; ++q) {
            const FxSide side = q < 2 ? fx_side_x(c[q]) : fx_side_y(c[q]);
            f[q] = q & 1 ? fx_flux_of<true>(c[q], side) : fx_flux_of<false>(c[q], side);
        }
        const FxSum s = dim == 1 ? fx_sum1(f[0], f[1]) : fx_sum2(f[0], f[1], f[2], f[3], 1, Split{});
        out[3 * k] = fx_value_E(s);
        out[3 * k + 1] = fx_value_X(s);
        out[3 * k + 2] = fx_value_Y(s);
    }
    return regular;
}

extern "C" int host_tail_blocks(int count) { return tail_blocks_for(count); }
