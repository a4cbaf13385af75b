// weak_rows.cuh -- writing a particle's rows for the weak pair kernels
// (kepler_weak.cuh): float4 [4][n].
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace sakura {

// component q of the position before the drift and of tau v
__device__ __forceinline__ void weak_row_component(float4 *rows, int64_t n, int64_t i, int q,
                                                   double x, double v, double tau)
{
    double *d = reinterpret_cast<double *>(rows);
    float *f = reinterpret_cast<float *>(rows);
    d[q < 2 ? 2 * i + q : 2 * (n + i)] = x;
    const double w = tau * v;
    const float h = __double2float_rn(w);
    f[4 * (2 * n + i) + q] = h;
    f[4 * (3 * n + i) + q] = __double2float_rn(w - (double)h);
}

// tau m and tau^2 m
__device__ __forceinline__ void weak_row_mass(float4 *rows, int64_t n, int64_t i, double m,
                                              double tau)
{
    double *d = reinterpret_cast<double *>(rows);
    float *f = reinterpret_cast<float *>(rows);
    const double mt = tau * m, mtt = tau * mt;
    d[2 * (n + i) + 1] = mt;
    const float h = __double2float_rn(mtt);
    f[4 * (2 * n + i) + 3] = h;
    f[4 * (3 * n + i) + 3] = __double2float_rn(mtt - (double)h);
}

}  // namespace sakura
