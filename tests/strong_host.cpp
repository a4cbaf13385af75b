// Host build of the conversions between double and double-word of the strong
// pairs (csrc/kepler_weak.cuh) for tests/test_strong_host.py.
#include "../paper_1402_3325_gb300/csrc/kepler_weak.cuh"

extern "C" void strong_split(long n, const double *x, float *h, float *l)
{
    for (long k = 0; k < n; ++k) {
        const sakura::dw s = sakura::dw_from_double(x[k]);
        h[k] = s.h;
        l[k] = s.l;
    }
}

extern "C" void strong_join(long n, const float *h, const float *l, double *out)
{
    for (long k = 0; k < n; ++k) out[k] = sakura::dw_double({h[k], l[k]});
}
