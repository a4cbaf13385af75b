// weak_rows.cuh -- writing a particle's rows for the weak pair kernels
// (kepler_weak.cuh): float4 [4][n]; and its three-float copy X3[20][n] for the
// double-word kernels that solve every pair (step_df64.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "df64.cuh"

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

// component q of the drifted position x and of the velocity v
__device__ __forceinline__ void tf_row_component(float *X3, int64_t n, int64_t i, int q, double x,
                                                 double v)
{
    float *p = X3 + 3 * q * n + i, *u = p + 9 * n;
    tf_split(x, p[0], p[n], p[2 * n]);
    tf_split(v, u[0], u[n], u[2 * n]);
}

__device__ __forceinline__ void tf_row_mass(float *X3, int64_t n, int64_t i, double m)
{
    const float h = __double2float_rn(m);
    X3[18 * n + i] = h;
    X3[19 * n + i] = __double2float_rn(m - (double)h);
}

}  // namespace sakura
