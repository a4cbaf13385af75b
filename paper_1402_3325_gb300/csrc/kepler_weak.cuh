// kepler_weak.cuh -- the order-2 pair map (Eq. 26) of a weakly perturbed pair
// to FP64 accuracy with few FP64 instructions.
//
// Why.  GB300 issues one FP64 warp instruction per 16 cycles per SM and 64
// FP32 ones in that time.  A seeded FP64 solve (kepler_fp64.cuh) takes 75
// FP64 instructions per pair and its kernels are bound by them.  Most pairs
// of a step move by a small part of their separation.  For those the map is
// a known leading term plus corrections, and only the leading term needs
// FP64 arithmetic: 16 FP64 instructions per pair, the corrections in
// double-word FP32 arithmetic (df64.cuh).
//
// In the units r0 (separation) and t (step), with x, w = t v the relative
// position before the step and the relative drift,
//   a = x.w / r0^2, b = w.w / r0^2, mu = m t^2 / r0^3, z = b - mu,
//   bt = beta t^2 / r0^2 = 2 mu - b, X = bt sigma^2,
//   sigma + a sigma^2 c2(X) + z sigma^3 c3(X) = 1      (universal Kepler),
//   rho = r / r0 = 1 + a sigma c1 + z sigma^2 c2,
// the increments of Eq. 26 are
//   delta_v / m = -(t / r0^3) [phi x + psi w],
//   delta_r / m = (t^2 / r0^3) [A x + B w],
//   phi = sigma c1 / rho = 1 + kappa, psi = sigma^2 c2 / rho,
//   A = phi / 2 - sigma^2 c2, B = psi / 2 - sigma^3 c3.
// |w| <= eps makes a = O(eps), and kappa, A and w itself too.  So
//   - x, r0^2, 1 / r0^3 (1 + kappa) and the sums of m x / r0^3 (1 + kappa)
//     are FP64;
//   - kappa, and everything that multiplies w or is multiplied by A, is a
//     double-word of about 2^-47 relative error, 2^-52 of the increment at
//     eps = 2^-5.  Quantities near 1 or 1/2 are held as their small
//     differences from it (u = sigma - 1, g1 = sigma c1 - 1, h2 = sigma^2 c2
//     - 1/2, p = rho - 1), which keeps that error relative to eps.
// sigma comes from one Newton step in single precision (error 2^-24) and
// one in double-word arithmetic, whose remainder is carried into c1, c2, c3
// and rho by their derivatives.
//
// x is the difference of the positions before the drift: the drifted and
// back-drifted difference of Eq. 17 without the two roundings.
//
// Which pairs (weak_class): |w| <= 2^-5 r0 and mu <= 2^-10, the speeds
// |t v_i|, |t v_j| below 2^-4 r0 (w is a difference of double-words, whose
// error is relative to them), all factors well inside float's range; every
// other pair takes the FP64 solve.  Up to that limit the velocity increments
// are no less accurate than the map in plain FP64 arithmetic (units of 2^-53
// r.m.s., here / plain FP64: 1.3 / 2.9 below 2^-9, 1.5 / 2.8 between 2^-7 and
// 2^-6, 1.8 / 2.9 up to 2^-5.5, 2.2 / 2.9 up to 2^-5;
// tests/test_weak_precision_host.py); the position's are off by 1.4 units of
// 2^-53 |t delta_v| / 2 at most.  A wider limit loses accuracy, a narrower
// one sends more pairs to the FP64 solve (their number grows with the limit's
// inverse cube: 0.7 % of the pairs of a 1024-body Plummer sphere at step
// 2^-8 with 2^-5, 5 % with 2^-6).
#pragma once

#include <cstdint>
#include <cstring>

#include "df64.cuh"
#include "fp_bits.cuh"


namespace sakura {

// -1/24, -1/120, 1/720 and 1/6 as double-words
constexpr float kWeakC24H = -0x1.555556p-5f;
constexpr float kWeakC24L = 0x1.555556p-30f;
constexpr float kWeakC120H = -0x1.111112p-7f;
constexpr float kWeakC120L = 0x1.dddddep-32f;
constexpr float kWeakC720H = 0x1.6c16c2p-10f;
constexpr float kWeakC720L = -0x1.27d27ep-35f;
constexpr float kWeakC6H = 0x1.555556p-3f;
constexpr float kWeakC6L = -0x1.555556p-28f;

// unnormalised double-word products and sums (|l| up to a few 2^-23 |h|)
DW_HD dw dwu_mul(dw x, dw y)
{
    const float p = fmul(x.h, y.h);
    const float e = ffma(x.h, y.h, -p);
    return {p, ffma(x.l, y.h, ffma(x.h, y.l, e))};
}
DW_HD dw dwu_mul_f(dw x, float y)
{
    const float p = fmul(x.h, y);
    return {p, ffma(x.l, y, ffma(x.h, y, -p))};
}
DW_HD dw dwu_add(dw x, dw y)
{
    const dw s = two_sum(x.h, y.h);
    return {s.h, fadd(s.l, fadd(x.l, y.l))};
}
DW_HD dw dwu_sub(dw x, dw y)
{
    const dw s = two_sum(x.h, -y.h);
    return {s.h, fadd(s.l, fsub(x.l, y.l))};
}
DW_HD dw dwu_norm(dw x) { return fast_two_sum(x.h, x.l); }

// a double in float range as h + l, h its leading 24 bits (truncated), l the
// next 23
DW_HD dw dw_split(double d)
{
#if defined(__CUDA_ARCH__)
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned t = __funnelshift_l(lo, hi, 3) ^ 0x40000000u;
    const unsigned hb = (t & 0x7fffffffu) | (hi & 0x80000000u);
    const unsigned eb = (hb & 0xff800000u) - (23u << 23);
    const float b = __uint_as_float(eb);
    const float c = __uint_as_float(eb + (((lo & 0x1fffffffu) + 32u) >> 6));
    return {__uint_as_float(hb), fsub(c, b)};
#else
    uint64_t u;
    std::memcpy(&u, &d, 8);
    const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
    const uint32_t t = ((hi << 3) | (lo >> 29)) ^ 0x40000000u;
    const uint32_t hb = (t & 0x7fffffffu) | (hi & 0x80000000u);
    const uint32_t eb = (hb & 0xff800000u) - (23u << 23);
    const uint32_t cb = eb + (((lo & 0x1fffffffu) + 32u) >> 6);
    float h, b, c;
    std::memcpy(&h, &hb, 4);
    std::memcpy(&b, &eb, 4);
    std::memcpy(&c, &cb, 4);
    return {h, fsub(c, b)};
#endif
}

// dw_split, 0 for |d| < 2^-100 (and for d = 0, which dw_split does not take)
DW_HD dw dw_split0(double d)
{
    const dw s = dw_split(d);
    const bool ok = ((uint32_t)((uint64_t)fpb_bits(d) >> 32) & 0x7ff00000u) >= 0x39b00000u;
    return {ok ? s.h : 0.0f, ok ? s.l : 0.0f};
}

// (double)f for a normal f on the integer pipe; a zero becomes 2^-127
DW_HD double widen(float f)
{
    const uint32_t u = fpb_fbits(f);
    return fpb_double((int64_t)((((uint64_t)(u & 0x80000000u)) << 32) |
                                (((uint64_t)(u & 0x7fffffffu) << 29) + (896ull << 52))));
}

// y^2 exactly (y > 0 normal), on the integer pipe
DW_HD double square_exact(float y)
{
    const uint32_t u = fpb_fbits(y);
    const uint32_t m = (u & 0x7fffffu) | 0x800000u;
    const uint64_t p = (uint64_t)m * m;  // in [2^46, 2^48)
    const uint32_t n = (uint32_t)(p >> 47);
    const uint32_t e = ((u >> 23) << 1) + n + 768u;
    return fpb_double((int64_t)((p << (6u - n)) + ((uint64_t)e << 52)));
}

// a b for normal a, b and a normal product, rounded to nearest even, on the
// integer pipe: the 106-bit product of the significands, normalised and
// rounded.
DW_HD double mul_soft(double a, double b)
{
    const uint64_t A = (uint64_t)fpb_bits(a), B = (uint64_t)fpb_bits(b);
    const uint32_t ah = (uint32_t)(A >> 32), al = (uint32_t)A;
    const uint32_t bh = (uint32_t)(B >> 32), bl = (uint32_t)B;
    const uint32_t ma = (ah & 0xfffffu) | 0x100000u, mb = (bh & 0xfffffu) | 0x100000u;
    const uint64_t L = (uint64_t)al * bl;
    const uint64_t W = (uint64_t)al * mb + ((uint64_t)ma * bl + (L >> 32));
    const uint64_t H = (uint64_t)ma * mb + (W >> 32);  // in [2^40, 2^42)
    const uint32_t wl = (uint32_t)W, hl = (uint32_t)H, hh = (uint32_t)(H >> 32);
    const uint32_t n = hh >> 9, sh = 12u - n;
    const uint32_t rh = (hh << sh) | (hl >> (32u - sh)), rl = (hl << sh) | (wl >> (32u - sh));
    // the bits below the significand: the upper one, and whether the rest is
    // more than nothing or the significand odd
    const uint32_t t = wl << sh;
    const uint32_t up = (t >> 31) & (uint32_t)(((t << 1) | (uint32_t)L | (rl & 1u)) != 0u);
    // the significand's hidden bit adds one to the exponent
    const uint32_t e = (ah & 0x7ff00000u) + (bh & 0x7ff00000u) + (n << 20) - (1024u << 20);
    const uint64_t r = (((uint64_t)(rh + e) << 32) | rl) + up;
    return fpb_double((int64_t)(r | ((uint64_t)((ah ^ bh) & 0x80000000u) << 32)));
}

// h + l as a double for |h| < 2^63; an exact zero stays zero, and so does the
// value of a subnormal float (the sums of light pairs end there): the floats
// are scaled by 2^64 into the normal range, on the FP32 pipe
DW_HD double dw_to_double(dw x)
{
    const float hs = fmul(x.h, 0x1p64f), ls = fmul(x.l, 0x1p64f);
    const int64_t down = 64LL << 52;
    const double h = fpb_double(fpb_bits(widen(hs)) - down);
    const double l = fpb_double(fpb_bits(widen(ls)) - down);
    return (x.h != 0.0f ? h : 0.0) + (x.l != 0.0f ? l : 0.0);
}

DW_HD float weak_float(uint32_t u)
{
#if defined(__CUDA_ARCH__)
    return __uint_as_float(u);
#else
    float f;
    std::memcpy(&f, &u, 4);
    return f;
#endif
}

// d as the nearest float and the float nearest to the rest, off the FP64 pipe
// (a conversion instruction costs as much as an FP64 one): |d| in [2^-126,
// 2^127); below, 0; above, infinity (NaN too).
DW_HD dw dw_from_double(double d)
{
    const uint64_t u = (uint64_t)fpb_bits(d), r = u + (1u << 28);
    const uint32_t hi = (uint32_t)(u >> 32), he = hi & 0x7ff00000u, sign = hi & 0x80000000u;
    if (!(he - 0x38100000u < 0x47e00000u - 0x38100000u))
        return {he < 0x38100000u ? 0.0f : weak_float(0x7f800000u), 0.0f};
    const uint32_t h = (((uint32_t)(r >> 29) ^ 0x40000000u) & 0x7fffffffu) | sign;
    // +-2^e of the exponent, and the 29 bits below h's as a signed integer
    const float e = weak_float((((hi << 3) ^ 0x40000000u) & 0x7f800000u) | sign);
    const float l = (float)(int32_t)((uint32_t)u << 3);
    return {weak_float(h), fmul(fmul(l, 0x1p-55f), e)};
}

// h + l as a double, off the FP64 pipe but for the sum
DW_HD double dw_double(dw x) { return f2d(x.h) + f2d(x.l); }

// Part of a pair's increments that do not depend on which particle takes
// them: Q (FP64) multiplies the separation, K the small terms.
struct WeakPair {
    double Q;             // (1 + kappa) / r0^3
    dw K, psi, Ap, Bp;    // 1 / r0^3, psi, A, B
};

// x: r_i - r_j before the drift, given as its double-word split xd and r2 =
// |x|^2 (split: r2d); w = tau (v_i - v_j); M = tau^2 (m_i + m_j)
DW_HD void weak_solve(double r2, dw r2d, const dw xd[3], const dw w[3], dw M, WeakPair &o)
{
    // y ~ 1/r0, e = 1 - r2 y^2
    float y = rsqrt_approx(r2d.h);
    {
        const float yy = fmul(y, y);
        y = ffma(fmul(0.5f, y), ffma(-r2d.l, yy, ffma(-r2d.h, yy, 1.0f)), y);
    }
    const double yd = widen(y);
    const double y2d = square_exact(y);
    const dw e = dw_split0(fma(-r2, y2d, 1.0));
    const dw p = two_prod(y, y);
    // a' = x.w, b' = w.w
    dw ap, bp;
    {
        const dw t0 = dwu_mul(xd[0], w[0]), t1 = dwu_mul(xd[1], w[1]), t2 = dwu_mul(xd[2], w[2]);
        ap = dwu_norm(dwu_add(dwu_add(t0, t1), t2));
        const dw s0 = dwu_mul(w[0], w[0]), s1 = dwu_mul(w[1], w[1]), s2 = dwu_mul(w[2], w[2]);
        bp = dwu_add(dwu_add(s0, s1), s2);
    }
    // 1/r0^2 = p (1 + e + e^2), 1/r0^3 = y p (1 + 3e/2 + 15e^2/8)
    const float ef = e.h;
    const dw i2 = fast_two_sum(p.h, ffma(p.h, ffma(ef, ef, ef), p.l));
    const dw yp = dwu_mul_f(p, y);
    const dw K = fast_two_sum(yp.h, ffma(yp.h, fmul(ef, ffma(1.875f, ef, 1.5f)), yp.l));
    const dw a = dwu_norm(dwu_mul(ap, i2));
    const dw b = dwu_mul(bp, i2);
    const dw mu = dwu_mul(M, K);
    const dw z = dwu_sub(b, mu);
    const dw bt = dwu_sub(mu, z);  // beta t^2 / r0^2
    // float root of sigma + a sigma^2 c2 + z sigma^3 c3 = 1
    float um;
    {
        const float u0 = ffma(a.h, ffma(0.5f, a.h, -0.5f), fmul(-1.0f / 6.0f, z.h));
        const float s = fadd(1.0f, u0);
        const float s2 = fmul(s, s);
        const float c2 = ffma(fmul(bt.h, s2), -1.0f / 24.0f, 0.5f);
        const float c3 = ffma(fmul(bt.h, s2), -1.0f / 120.0f, 1.0f / 6.0f);
        const float t2 = fmul(s2, c2), t3 = fmul(fmul(s2, s), c3);
        const float F = ffma(z.h, t3, ffma(a.h, t2, u0));
        const float Fp = ffma(z.h, t2, ffma(a.h, s, 1.0f));
        um = ffma(-F, rcp_approx(Fp), u0);
    }
    const float sg = fadd(1.0f, um);
    um = fsub(sg, 1.0f);  // exact
    const dw q2 = two_prod(sg, sg);
    const dw X = dwu_mul(bt, q2);
    const float Xf = X.h;
    // k2 = c2 - 1/2, c3, k1 = c1 - 1
    const dw k2t = dwu_mul(X, dw{kWeakC720H, ffma(Xf, -1.0f / 40320.0f, kWeakC720L)});
    dw g2 = fast_two_sum(kWeakC24H, k2t.h);
    g2.l = fadd(g2.l, fadd(k2t.l, kWeakC24L));
    const dw k2 = dwu_mul(X, g2);
    const dw c3t = dwu_mul(X, dw{kWeakC120H, ffma(Xf, ffma(Xf, -1.0f / 362880.0f, 1.0f / 5040.0f), kWeakC120L)});
    dw c3 = fast_two_sum(kWeakC6H, c3t.h);
    c3.l = fadd(c3.l, fadd(c3t.l, kWeakC6L));
    const dw nk1 = dwu_mul(X, c3);  // -k1
    // h2 = sigma^2 c2 - 1/2
    const dw uu = two_prod(um, um);
    const dw s2k2 = dwu_mul(q2, k2);
    dw h2 = fast_two_sum(um, fmul(0.5f, uu.h));
    h2.l = ffma(0.5f, uu.l, h2.l);
    h2 = dwu_add(h2, s2k2);
    // g1 = sigma c1 - 1
    const dw sk1 = dwu_mul_f(nk1, sg);
    dw g1 = two_sum(um, -sk1.h);
    g1.l = fsub(g1.l, sk1.l);
    const dw s3c3 = dwu_mul(dwu_mul_f(q2, sg), c3);
    // F and p = rho - 1 at sigma
    const dw ah2 = dwu_mul(a, h2);
    const dw T2 = dwu_mul(z, s3c3);
    const dw zh2 = dwu_mul(z, h2);
    const dw ag1 = dwu_mul(a, g1);
    dw F = two_sum(um, fmul(0.5f, a.h));
    F.l = ffma(0.5f, a.l, F.l);
    F = dwu_add(F, dwu_add(ah2, T2));
    dw pr = two_sum(a.h, fmul(0.5f, z.h));
    pr.l = fadd(pr.l, ffma(0.5f, z.l, a.l));
    pr = dwu_norm(dwu_add(pr, dwu_add(ag1, zh2)));
    // delta = F / (1 + p)
    float ir = rcp_approx(fadd(1.0f, pr.h));
    const float d1 = fmul(fadd(F.h, F.l), ir);
    const float rem = fadd(ffma(-d1, pr.h, fsub(F.h, d1)), F.l);
    const float d2 = fmul(rem, ir);
    // carry to the root
    const float xc2 = fmul(Xf, fadd(0.5f, k2.h));
    const float dX = fmul(d1, xc2);
    const float psi0 = fadd(0.5f, h2.h);
    h2 = dwu_add(h2, dw{-d1, ffma(d1, ffma(0.5f, d1, -g1.h), -d2)});
    pr.l = ffma(-d1, ffma(-a.h, xc2, ffma(z.h, g1.h, fadd(a.h, z.h))), pr.l);
    g1 = dwu_add(g1, dw{-d1, fsub(dX, d2)});
    // kappa = (g1 - p) / (1 + p)
    const dw N = dwu_norm(dwu_sub(g1, pr));
    const float k1 = fmul(N.h, ir);
    const float r1 = fadd(ffma(-k1, pr.h, fsub(N.h, k1)), ffma(-k1, pr.l, N.l));
    const float kl = fmul(r1, ir);
    // 1/rho
    const float rr = ffma(-ir, pr.l, ffma(-ir, pr.h, fsub(1.0f, ir)));
    const dw ip = {ir, fmul(ir, rr)};
    const dw hp = fast_two_sum(0.5f, h2.h);
    const dw psi = dwu_norm(dwu_mul(dw{hp.h, fadd(hp.l, h2.l)}, ip));
    // kappa' = (1 + kappa)(1 + 3e/2 + 15 e^2/8) - 1 as kp.h + kl', every
    // product above 2^-54 in it, and both parts into the FP64 factor: the
    // second one (up to 2^-28) as a term of the double-word sums instead, and
    // without the products of second parts, made the error along x 3.1 units
    // of 2^-53 r.m.s. where this is 2.3
    dw et = two_prod(1.5f, e.h);
    et.l = ffma(1.5f, e.l, ffma(et.h, fmul(1.25f, ef), et.l));
    const dw kp = two_sum(k1, et.h);
    const float kq = ffma(et.h, k1, fadd(kl, ffma(et.h, kl, ffma(et.l, k1, et.l))));
    const double y3 = y2d * yd;
    o.Q = fma(y3, widen(kp.h) + widen(fadd(kp.l, kq)), y3);
    o.K = K;
    o.psi = psi;
    o.Ap = dwu_norm(dwu_sub(dw{0.5f * k1, 0.5f * kl}, h2));
    const dw s3 = {s3c3.h, ffma(-d1, psi0, ffma(-0.5f, d2, s3c3.l))};
    o.Bp = dwu_norm(dwu_sub(dw{0.5f * psi.h, 0.5f * psi.l}, s3));
}

// acc += x y
DW_HD void weak_acc(dw &acc, dw x, dw y)
{
    const float p = fmul(x.h, y.h);
    const float e = ffma(x.l, y.h, ffma(x.h, y.l, ffma(x.h, y.h, -p)));
    const dw s = two_sum(acc.h, p);
    acc.h = s.h;
    acc.l = fadd(acc.l, fadd(s.l, e));
}

// the limits of weak_class, as ratios to r0^2 or plain
constexpr float kWeakEps2 = 0x1p-10f, kWeakMu = 0x1p-10f, kWeakSpeed2 = 0x1p-8f;
// Smallest tau^2 m / r0^2 of a particle, and smallest tau^2 m and tau^2 m /
// r0^3: a float's last place is no smaller than 2^-149, so the increments'
// double-word sums (of the size of the first times eps r0) are off by up to a
// few 2^-149, 2^-54 of the increment, and the remainders of the mass and of
// its product with 1 / r0^3 by 2^-50, times eps.
constexpr float kWeakMin = 1e-28f, kWeakMinFactor = 0x1p-100f;

// One particle: position before the drift, tau m, and tau v, tau^2 m as
// double-words.
struct WeakParticle {
    double x, y, z, mt;
    dw w[3], mh;
};

DW_HD float weak_speed2(const WeakParticle &p)
{
    return ffma(p.w[0].h, p.w[0].h, ffma(p.w[1].h, p.w[1].h, fmul(p.w[2].h, p.w[2].h)));
}

struct WeakDiff {
    double x[3], r2;
    dw r2d, w[3];
    float w2, y;  // |w|^2, 1 / r0
};

// Relative state of the pair and whether it takes weak_add (sa =
// weak_speed2(a)).  r0^2 in [2^-60, 2^60) is tested on its exponent field;
// NaN and infinities fail a test and go to the FP64 solve, which reports
// them.
DW_HD bool weak_class(const WeakParticle &a, float sa, const WeakParticle &b, WeakDiff &d)
{
    d.x[0] = a.x - b.x;
    d.x[1] = a.y - b.y;
    d.x[2] = a.z - b.z;
    d.r2 = fma(d.x[0], d.x[0], fma(d.x[1], d.x[1], d.x[2] * d.x[2]));
    const uint32_t hi = (uint32_t)((uint64_t)fpb_bits(d.r2) >> 32);
    d.r2d = dw_split(d.r2);
    for (int q = 0; q < 3; ++q) {
        const dw s = two_sum(a.w[q].h, -b.w[q].h);
        d.w[q] = fast_two_sum(s.h, fadd(s.l, fsub(a.w[q].l, b.w[q].l)));
    }
    d.w2 = ffma(d.w[0].h, d.w[0].h, ffma(d.w[1].h, d.w[1].h, fmul(d.w[2].h, d.w[2].h)));
    d.y = rsqrt_approx(d.r2d.h);
    const float y2 = fmul(d.y, d.y);
    const float mu = fmul(fmul(fadd(a.mh.h, b.mh.h), d.y), y2), mm = fminf(a.mh.h, b.mh.h);
    return hi - 0x3c300000u < 0x07800000u && d.w2 <= fmul(kWeakEps2, d.r2d.h) &&
           fadd(sa, weak_speed2(b)) <= fmul(kWeakSpeed2, d.r2d.h) && mu <= kWeakMu &&
           fmul(mm, y2) >= kWeakMin && fmul(mm, fminf(1.0f, fmul(d.y, y2))) >= kWeakMinFactor;
}

// Whether a class test of e < e_max < 1 on float copies (kepler_fp32.cuh) is
// certain to find the pair unbound, (v^2 - 2 m / r0) h^2 >= 0: v^2 above 2 m
// / r0 and h^2 = r0^2 v^2 - (r0.v)^2 above 0, each by more than the test's
// roundings: of v^2 up to 2^-22 |v| (|v_i| + |v_j|), which is at most 2^-10
// v^2 + 2^-32 (v_i^2 + v_j^2), and of h^2 up to 2^-21 r0^2 v^2.
DW_HD bool weak_unbound(const WeakParticle &a, float sa, const WeakParticle &b, const WeakDiff &d)
{
    const float pot = fmul(fmul(2.0f * 1.004f, fadd(a.mh.h, b.mh.h)), d.y);
    const float x = dw_split0(d.x[0]).h, y = dw_split0(d.x[1]).h, z = dw_split0(d.x[2]).h;
    const float xw = ffma(x, d.w[0].h, ffma(y, d.w[1].h, fmul(z, d.w[2].h)));
    return fmul(d.w2, 0.998f) > ffma(fadd(sa, weak_speed2(b)), 0x1p-30f, pot) &&
           fmul(xw, xw) < fmul(1.0f - 0x1p-16f, fmul(d.w2, d.r2d.h));
}

// Adds the pair's increments to the sums of both particles:
//   vr, vc: the velocity terms along x, FP64, final units;
//   er, ec: the other velocity terms, to be scaled by -1/tau;
//   rr, rc: position.
// The column's sums keep the row's sign (the caller negates them).
DW_HD void weak_add(const WeakParticle &a, const WeakParticle &b, const WeakDiff &d,
                    double vr[3], dw er[3], dw rr[3], double vc[3], dw ec[3], dw rc[3])
{
    const dw xd[3] = {dw_split0(d.x[0]), dw_split0(d.x[1]), dw_split0(d.x[2])};
    WeakPair o;
    weak_solve(d.r2, d.r2d, xd, d.w, dwu_add(a.mh, b.mh), o);
    // on the integer pipe (about 25 instructions): 3 % of a step on tiles at
    // 4000 bodies, 1 % in row groups at 16384.  The other two multiplies (y^3,
    // z^2) there too gained nothing more.
    const double qj = mul_soft(b.mt, o.Q), qi = mul_soft(a.mt, o.Q);
    for (int q = 0; q < 3; ++q) {
        vr[q] = fma(-qj, d.x[q], vr[q]);
        vc[q] = fma(-qi, d.x[q], vc[q]);
    }
    const dw Kj = dwu_mul(b.mh, o.K), Ki = dwu_mul(a.mh, o.K);
    for (int q = 0; q < 3; ++q) {
        const dw e = dwu_mul(o.psi, d.w[q]);
        weak_acc(er[q], Kj, e);
        weak_acc(ec[q], Ki, e);
        const dw r = dwu_add(dwu_mul(o.Ap, xd[q]), dwu_mul(o.Bp, d.w[q]));
        weak_acc(rr[q], Kj, r);
        weak_acc(rc[q], Ki, r);
    }
}

#if defined(__CUDACC__)
// A particle's four 16-byte rows (weak_rows.cuh): (x, y) and (z, tau m) as
// doubles, the leading floats of (tau vx, tau vy, tau vz, tau^2 m) and their
// remainders.
__device__ __forceinline__ WeakParticle weak_unpack(const float4 &a, const float4 &b,
                                                    const float4 &h, const float4 &l)
{
    WeakParticle p;
    p.x = __hiloint2double(__float_as_int(a.y), __float_as_int(a.x));
    p.y = __hiloint2double(__float_as_int(a.w), __float_as_int(a.z));
    p.z = __hiloint2double(__float_as_int(b.y), __float_as_int(b.x));
    p.mt = __hiloint2double(__float_as_int(b.w), __float_as_int(b.z));
    p.w[0] = {h.x, l.x};
    p.w[1] = {h.y, l.y};
    p.w[2] = {h.z, l.z};
    p.mh = {h.w, l.w};
    return p;
}
#endif

}  // namespace sakura
