// Host entries to the kernels' arithmetic that is host code too (m1_fx.cuh,
// m1_strip64.cuh), for tests that need no GPU (tests/fx_host.py compiles this file).
#include "m1_strip64.cuh"

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
