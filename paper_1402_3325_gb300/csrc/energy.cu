// energy.cu -- total energy E = T + U of a device state (Eqs. 1-3).
//
// Stage 1: rows r and n-1-r have n - 1 pairs (j > i) between them; the list
// of these row pairs, each cut into S equal segments, is dealt to the warps,
// lanes stride over j.  A lane sums m_j / r_ij of four pairs and adds the sum
// to a double-double (Fast2Sum, Dekker 1971, of the operands in order of
// size); the row's factor -m_i is applied once per row, in double-double.
// Warps reduce their lanes in double-double and write one (hi, lo) pair each.
// Stage 2: one block adds the kinetic terms m_i v_i^2 / 2 and the warp
// partials in a fixed order, in double-double, and writes E and the status
// word to page-locked host memory (a copy-engine read costs about 10 us more
// per call).  No atomics on FP64 data; the result does not depend on timing.
//
// Bound: the FP64 pipe, 10.5 instructions per pair at 16 cycles per warp
// instruction and SM (2.4 ms at 16384 bodies).  1/r comes from a
// single-precision value y by one Newton step in FP64, 1/r = y (1 + e/2 +
// 3 e^2/8), e = 1 - r^2 y^2 with y^2 exact on the integer pipe; the last
// term, below 2^-43 of the value, is summed in single precision.  With sqrt,
// a division and a six-operation TwoSum per pair it took 7.96 ms.
#include <cuda_runtime.h>

#include "kepler_fp64.cuh"
#include "kepler_weak.cuh"
#include "step_common.cuh"

namespace sakura {
namespace {

constexpr int kEnergyThreads = 256;
constexpr int kEnergyBlocks = 152 * 3;

__device__ __forceinline__ void dd_add(double &s, double &c, double x)
{
    const double t = s + x;
    const double bp = t - s;
    const double e = (s - (t - bp)) + (x - bp);
    s = t;
    c += e;
}

__device__ __forceinline__ void dd_merge(double &s, double &c, double s2, double c2)
{
    dd_add(s, c, s2);
    c += c2;
}

// s + c += x, c the sum of the rounding errors
__device__ __forceinline__ void dd_add_ordered(double &s, double &c, double x)
{
    const bool swap = magbits(x) > magbits(s);
    const double big = swap ? x : s, sml = swap ? s : x;
    s = big + sml;
    c += sml - (s - big);
}

// m / sqrt(r2); the term below 2^-43 of it goes to lo, in single precision,
// where the value is in float's range
__device__ __forceinline__ double inv_distance(double r2, double m, float &lo)
{
    const long long b = dbits(r2);
    // outside [2^-120, 2^120): zero (reported by the caller), subnormal,
    // overflown or not a number
    if (!((unsigned long long)b - 0x3870000000000000ULL < 0x0f00000000000000ULL))
        return m / sqrt(r2);
    const float y = rsqrt_approx(trunc_to_f32(b));
    // e / 2 = 1/2 - (r2 / 2) y^2
    const double eh = fma(-__longlong_as_double(b - (1LL << 52)), square_exact(y), 0.5);
    const double t = m * widen_f32(y);
    const long long bt = dbits(t), be = dbits(eh);
    if ((bt & kInfBits) - 0x39b0000000000000LL < 0x0c80000000000000LL &&
        (bt & kInfBits) >= 0x39b0000000000000LL) {  // 2^-100 <= |t| < 2^100
        const float ef = (be & kInfBits) >= 0x39b0000000000000LL ? trunc_to_f32(be) : 0.0f;
        lo = fmaf(1.5f * ef * ef, trunc_to_f32(bt), lo);
        return fma(t, eh, t);
    }
    return fma(t, fma(1.5 * eh, eh, eh), t);
}

// -m_i sum_j m_j / r_ij over j0 <= j < j1 (this lane's), added to (s, c)
__device__ __forceinline__ void row_potential(const double *state, const double *mass, int64_t n,
                                              int64_t i, int64_t j0, int64_t j1, int lane,
                                              double &s, double &c, unsigned &st)
{
    const double xi = state[i], yi = state[n + i], zi = state[2 * n + i], mi = mass[i];
    double us = 0.0, uc = 0.0;
    float lo = 0.0f;
    auto term = [&](int64_t j) {
        const double dx = xi - state[j], dy = yi - state[n + j], dz = zi - state[2 * n + j];
        const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
        if (!(dbits(r2) > 0 && dbits(r2) <= kInfBits)) st |= kStatusCoincident;
        return inv_distance(r2, mass[j], lo);
    };
    int64_t j = j0 + lane;
    for (; j + 96 < j1; j += 128) {
        const double a = term(j), b = term(j + 32), d = term(j + 64), e = term(j + 96);
        dd_add_ordered(us, uc, (a + b) + (d + e));
    }
    for (; j < j1; j += 32) dd_add_ordered(us, uc, term(j));
    uc += (double)lo;
    const double p = -mi * us;
    dd_add(s, c, p);
    c += fma(-mi, us, -p) - mi * uc;
}

__global__ void __launch_bounds__(kEnergyThreads, 3)
    energy_pairs_kernel(const double *state, const double *mass, int64_t n, int S, double *work,
                        unsigned *status)
{
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t W = ((int64_t)gridDim.x * blockDim.x) >> 5;
    double s = 0.0, c = 0.0;
    unsigned st = 0;
    const int64_t half = (n + 1) / 2;
    for (int64_t q = w; q < half * S; q += W) {
        // segment k of the n - 1 pairs of rows r and n - 1 - r
        const int64_t r = q / S, k = q - r * S;
        const int64_t a = k * (n - 1) / S, b = (k + 1) * (n - 1) / S, first = n - 1 - r;
        const int64_t r2 = n - 1 - r;
        if (a < first)
            row_potential(state, mass, n, r, r + 1 + a, r + 1 + (b < first ? b : first), lane, s,
                          c, st);
        if (b > first && r2 != r)
            row_potential(state, mass, n, r2, r2 + 1 + (a > first ? a - first : 0),
                          r2 + 1 + b - first, lane, s, c, st);
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double s2 = __shfl_xor_sync(0xffffffffu, s, o);
        const double c2 = __shfl_xor_sync(0xffffffffu, c, o);
        // combine in a lane-order-independent way: the lower lane id keeps its
        // own value first, so both partners compute the same bits
        if ((lane & o) == 0) {
            dd_merge(s, c, s2, c2);
        } else {
            double a = s2, b = c2;
            dd_merge(a, b, s, c);
            s = a;
            c = b;
        }
    }
    st = __reduce_or_sync(0xffffffffu, st);
    if (lane == 0) {
        work[w] = s;
        work[W + w] = c;
        if (st) atomicOr(status, st);
    }
}

__global__ void __launch_bounds__(1024)
    energy_final_kernel(const double *state, const double *mass, int64_t n, const double *work,
                        int64_t W, double *out, unsigned *status, unsigned *host_status)
{
    __shared__ double sh_s[1024], sh_c[1024], sh_t[1024], sh_tc[1024];
    const int t = threadIdx.x;
    double ks = 0.0, kc = 0.0, us = 0.0, uc = 0.0;
    for (int64_t i = t; i < n; i += blockDim.x) {
        const double vx = state[3 * n + i], vy = state[4 * n + i], vz = state[5 * n + i];
        dd_add(ks, kc, 0.5 * mass[i] * fma(vx, vx, fma(vy, vy, vz * vz)));
    }
    for (int64_t w = t; w < W; w += blockDim.x) dd_merge(us, uc, work[w], work[W + w]);
    sh_s[t] = us;
    sh_c[t] = uc;
    sh_t[t] = ks;
    sh_tc[t] = kc;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (t < h) {
            double a = sh_s[t], b = sh_c[t];
            dd_merge(a, b, sh_s[t + h], sh_c[t + h]);
            sh_s[t] = a;
            sh_c[t] = b;
            double p = sh_t[t], q = sh_tc[t];
            dd_merge(p, q, sh_t[t + h], sh_tc[t + h]);
            sh_t[t] = p;
            sh_tc[t] = q;
        }
        __syncthreads();
    }
    if (t == 0) {
        double es = 0.0, ec = 0.0;
        dd_merge(es, ec, sh_t[0], sh_tc[0]);
        dd_merge(es, ec, sh_s[0], sh_c[0]);
        out[0] = es + ec;
        out[1] = sh_t[0] + sh_tc[0];
        out[2] = sh_s[0] + sh_c[0];
        const unsigned st = *status;
        *host_status = st;
        if (st) *status = 0u;
    }
}

}  // namespace

int energy_work_size(int64_t n)
{
    (void)n;
    return 2 * kEnergyBlocks * (kEnergyThreads / 32);
}

void launch_energy(const double *state, const double *mass, int64_t n, double *work, double *out,
                   unsigned *status, unsigned *host_status, cudaStream_t s)
{
    // segments of about 1024 pairs or more, so that the last round of the
    // warps is short; no more blocks than there are segments for
    const int S = (int)(n < 2048 ? 1 : (n < 8192 ? n / 1024 : 8));
    const int64_t items = (n + 1) / 2 * S, per = kEnergyThreads / 32;
    const int64_t need = (items + per - 1) / per;
    const int blocks = (int)(need < kEnergyBlocks ? need : kEnergyBlocks);
    energy_pairs_kernel<<<blocks, kEnergyThreads, 0, s>>>(state, mass, n, S, work, status);
    energy_final_kernel<<<1, 1024, 0, s>>>(state, mass, n, work, blocks * per, out, status,
                                           host_status);
}

}  // namespace sakura
