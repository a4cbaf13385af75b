// kepler_weak32.cuh -- the FP32-class pairs of the mixed-precision form that
// move little in the step (nearly all of them): the pair map of Eq. 26 in
// FP32 without the iteration of kepler_fp32.cuh.
//
// With x, v, m the pair's Kepler input, t the step, in the units r0 and t,
//   a = x.v t / r0^2, b = v.v t^2 / r0^2, mu = m t^2 / r0^3, z = b - mu,
//   Y = (2 mu - b) sigma^2,
//   sigma + a sigma^2 c2(Y) + z sigma^3 c3(Y) = 1     (universal Kepler),
//   rho = r / r0 = 1 + a sigma c1 + z sigma^2 c2,
// the increments are
//   delta_v / m = -(t / r0^3) [phi x + psi t v],
//   delta_r / m = (t^2 / r0^3) [(post phi - g2) x + (post psi - g3) t v],
//   g_k = sigma^k c_k, phi = g1 / rho, psi = g2 / rho.
// b <= 2^-8 and mu <= 2^-8 make |a| <= 2^-4 and |Y| < 2^-7.  So two terms
// of c2 and c3 reach 2^-24 of them (the third is Y^2 / 360 < 2^-22.4 of c2,
// kept; Y^2 / 840 < 2^-23.7 of c3, whose weight in the increments is b, mu or
// less), the second-order root 1 - a / 2 + a^2 / 2 - z / 6 is within 2^-11,
// and one Newton step, carried through g1, g2, g3 and rho by their
// derivatives, leaves 2^-25.  Every quantity is a float as in kepler_fp32.cuh;
// phi and rho enter by their small differences from 1.  The error measured
// against the exact map, in units of 2^-24 of the velocity increment and of
// |t delta_v| / 2 for the position's, r.m.s. over b from 2^-24 to the limit,
// with roots up to one unit off as the hardware's are: 1.2 and 1.4, where the
// iteration of kepler_fp32.cuh has 2.3 and 1.7 (worst of 900000 pairs 5.7 and
// 6.1 against 10.4 and 9.2).  The last three conditions keep
// separations and increments far from float's overflow.
#pragma once

#include "df64.cuh"

namespace sakura {

constexpr float kWeak32Max = 0x1p-8f;  // the limit of b and of mu

// The increments divided by m (out[0..2] position, out[3..5] velocity) and
// whether the pair is within the limits; for others out has no meaning.
DW_HD bool pair32_weak(const float x[3], const float v[3], float r2, float v2, float eta, float m,
                       float ir0, float tau, float post, float out[6])
{
    const float ti = fmul(tau, ir0), ti2 = fmul(ti, ti);
    const float b = fmul(v2, ti2), mu = fmul(fmul(m, ir0), ti2);
    const float a = fmul(fmul(eta, ir0), ti);
    const float z = fsub(b, mu), bt = ffma(2.0f, mu, -b);
    // u = sigma - 1
    const float u = ffma(a, ffma(0.5f, a, -0.5f), fmul(-1.0f / 6.0f, z));
    const float s = fadd(1.0f, u), s2 = fmul(s, s);
    const float Y = fmul(bt, s2);
    const float c2 = ffma(Y, ffma(Y, 1.0f / 720.0f, -1.0f / 24.0f), 0.5f);
    const float c3 = ffma(Y, -1.0f / 120.0f, 1.0f / 6.0f);
    const float c0 = ffma(-Y, c2, 1.0f);
    const float e1 = ffma(-fmul(Y, c3), s, u);  // g1 - 1
    const float g1 = fadd(1.0f, e1), g2 = fmul(s2, c2), g3 = fmul(fmul(s2, s), c3);
    const float F = ffma(a, g2, ffma(z, g3, u));
    const float p = ffma(a, g1, fmul(z, g2));  // rho - 1
    const float d = fmul(-F, rcp_approx(fadd(1.0f, p)));
    const float h2 = ffma(d, ffma(0.5f, fmul(d, c0), g1), g2);
    const float h3 = ffma(d, g2, g3);
    const float pr = ffma(d, ffma(a, c0, fmul(z, g1)), p);
    const float ir = rcp_approx(fadd(1.0f, pr));
    const float phi1 = fmul(fsub(ffma(d, c0, e1), pr), ir);  // phi - 1
    const float psi = fmul(h2, ir);
    // t / r0^3 from the approximate root ir0, whose error the leading term
    // carries three times: (1 - r0^2 ir0^2) 3 / 2 corrects it
    const float y2 = fmul(ir0, ir0), k = fmul(ti, y2), kt = fmul(ti2, ir0);
    const float vx = ffma(-k, ffma(1.5f, ffma(-r2, y2, 1.0f), phi1), -k), vv = -fmul(kt, psi);
    const float rx = fmul(kt, ffma(post, fadd(1.0f, phi1), -h2));
    const float rv = fmul(fmul(kt, tau), ffma(post, psi, -h3));
    for (int q = 0; q < 3; ++q) {
        out[q] = ffma(rx, x[q], fmul(rv, v[q]));
        out[3 + q] = ffma(vx, x[q], fmul(vv, v[q]));
    }
    return b <= kWeak32Max && mu <= kWeak32Max && ir0 >= 0x1p-62f && fabsf(k) <= 0x1p60f &&
           kt <= 0x1p60f;
}

}  // namespace sakura
