// Host build of the FP32 weak pair map (csrc/kepler_weak32.cuh) for the CPU
// test of its accuracy.
#include "../paper_1402_3325_gb300/csrc/kepler_weak32.cuh"

#include <cmath>

using namespace sakura;

extern "C" void weak32(long n, const float *x, const float *v, const float *m, const float *tau,
                       float post, int *weak, float *out)
{
    for (long k = 0; k < n; ++k) {
        const float *a = x + 3 * k, *b = v + 3 * k;
        const float r2 = ffma(a[0], a[0], ffma(a[1], a[1], a[2] * a[2]));
        const float v2 = ffma(b[0], b[0], ffma(b[1], b[1], b[2] * b[2]));
        const float eta = ffma(a[0], b[0], ffma(a[1], b[1], a[2] * b[2]));
        // a root one unit off, as the hardware's approximation may be
        float ir0 = (float)(1.0 / std::sqrt((double)r2));
        if (r2 > 0.0f && k % 3) ir0 = std::nextafterf(ir0, k % 3 == 1 ? 0.0f : INFINITY);
        weak[k] = pair32_weak(a, b, r2, v2, eta, m[k], ir0, tau[k], post, out + 6 * k);
    }
}
