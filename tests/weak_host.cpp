// Host build of the weak pair map (csrc/kepler_weak.cuh) for the CPU test of
// its accuracy (tests/test_weak_host.py).  Built with -ffp-contract=off so
// that every float operation rounds once.
#include "../paper_1402_3325_gb300/csrc/kepler_weak.cuh"

using namespace sakura;

static dw to_dw(double d)
{
    const float h = (float)d;
    return {h, (float)(d - (double)h)};
}

static WeakParticle particle(const double *r, const double *v, double m, double tau)
{
    WeakParticle p;
    p.x = r[0];
    p.y = r[1];
    p.z = r[2];
    p.mt = tau * m;
    for (int q = 0; q < 3; ++q) p.w[q] = to_dw(tau * v[q]);
    p.mh = to_dw(tau * p.mt);
    return p;
}

// For each pair k of particles (ri, vi, mi), (rj, vj, mj): whether it is weak
// and, if so, the increments it adds to i and to j (positions, velocities),
// as leading and remaining part.
extern "C" void weak_pairs(long n, const double *ri, const double *vi, const double *mi,
                           const double *rj, const double *vj, const double *mj, double tau,
                           int *weak, double *inc, double *rest)
{
    for (long k = 0; k < n; ++k) {
        const WeakParticle a = particle(ri + 3 * k, vi + 3 * k, mi[k], tau);
        const WeakParticle b = particle(rj + 3 * k, vj + 3 * k, mj[k], tau);
        WeakDiff d;
        weak[k] = weak_class(a, weak_speed2(a), b, d);
        if (!weak[k]) continue;
        double vr[3] = {0, 0, 0}, vc[3] = {0, 0, 0};
        dw er[3], rr[3], ec[3], rc[3];
        for (int q = 0; q < 3; ++q) er[q] = rr[q] = ec[q] = rc[q] = dw{0.0f, 0.0f};
        weak_add(a, b, d, vr, er, rr, vc, ec, rc);
        for (int q = 0; q < 3; ++q) {
            inc[12 * k + q] = dw_to_double(rr[q]);
            inc[12 * k + 3 + q] = vr[q];
            inc[12 * k + 6 + q] = -dw_to_double(rc[q]);
            inc[12 * k + 9 + q] = -vc[q];
            rest[12 * k + q] = rest[12 * k + 6 + q] = 0.0;
            rest[12 * k + 3 + q] = -dw_to_double(er[q]) / tau;
            rest[12 * k + 9 + q] = dw_to_double(ec[q]) / tau;
        }
    }
}

extern "C" void weak_squares(long n, const float *y, double *out)
{
    for (long k = 0; k < n; ++k) out[k] = square_exact(y[k]);
}

extern "C" void weak_splits(long n, const double *x, double *out)
{
    for (long k = 0; k < n; ++k) {
        const dw s = dw_split0(x[k]);
        out[k] = (double)s.h + (double)s.l;
    }
}

extern "C" void weak_products(long n, const double *a, const double *b, double *out)
{
    for (long k = 0; k < n; ++k) out[k] = mul_soft(a[k], b[k]);
}
