"""CPU check of the weak pair map (csrc/kepler_weak.cuh) for light particles
and extreme separations: whatever pair the class test admits, its increments
are as accurate as those of ordinary ones."""
import numpy as np
import pytest

mpmath = pytest.importorskip("mpmath")

from test_weak_host import U, _exact, _run, lib  # noqa: E402,F401


def _pairs(log_r, log_m, eps, n=40):
    """n pairs at separations near 2^log_r that move by eps of it in a step
    of 2^-8, tau^2 m / r0^2 = 2^log_m."""
    rng = np.random.default_rng(1000 - log_m + log_r)
    unit = lambda: (lambda a: a / np.linalg.norm(a, axis=1)[:, None])(rng.normal(size=(n, 3)))
    tau, r0 = 2.0 ** -8, 2.0 ** log_r * np.exp(rng.uniform(-0.3, 0.3, n))
    x, w = unit() * r0[:, None], unit() * (eps * r0)[:, None]
    m, part = 2.0 ** log_m * r0 ** 2 / tau ** 2, rng.uniform(0.2, 0.8, n)
    c, f = rng.normal(size=(n, 3)) * r0[:, None], (1 - part)[:, None]
    return (c + f * x, f * w / tau, part * m, c - (1 - f) * x, -(1 - f) * w / tau, (1 - part) * m,
            tau)


# the bounds of test_weak_map_against_the_exact_one (a cold pair's correction
# is mu, below 2^-12 here), and one double-word's last places more: the sums
# end at 2^-149, 2^-54 of an increment at the class's limit, twice over in a
# pair's three components
@pytest.mark.parametrize("eps,bound_v,bound_r", [(0.0, 2.5, 1.0), (2.0 ** -30, 2.5, 1.0),
                                                 (2.0 ** -12, 2.5, 1.0), (2.0 ** -6, 6.5, 4.5)])
@pytest.mark.parametrize("log_r,log_m,admitted", [
    (0, -90, True), (0, -80, True), (0, -72, True), (-10, -90, False), (-10, -75, True),
    (-29, -80, False), (-29, -50, False), (-29, -40, False), (29, -90, False), (29, -80, False),
    (29, -66, True)])
def test_light_pairs_are_accurate_or_left_to_the_general_solve(lib, log_r, log_m, admitted, eps,  # noqa: F811
                                                               bound_v, bound_r):
    ri, vi, mi, rj, vj, mj, tau = _pairs(log_r, log_m, eps)
    weak, inc, rest = _run(lib, ri, vi, mi, rj, vj, mj, tau)
    assert weak.mean() > 0.7 if admitted else True
    ev, er = [0.0], [0.0]
    for k in np.flatnonzero(weak):
        with mpmath.workdps(60):
            f = mpmath.mpf
            dr, dv = _exact(ri[k], vi[k], rj[k], vj[k], f(mi[k]) + f(mj[k]), tau)
            nv = mpmath.sqrt(sum(q * q for q in dv))
            for side, mass in ((0, f(mj[k])), (6, -f(mi[k]))):
                got = [f(inc[k, side + q]) + f(rest[k, side + q]) for q in range(6)]
                ev.append(float(mpmath.sqrt(sum((got[3 + q] - mass * dv[q]) ** 2
                                                for q in range(3))) / (abs(mass) * nv)) / U)
                er.append(float(mpmath.sqrt(sum((got[q] - mass * dr[q]) ** 2 for q in range(3)))
                                / (abs(mass) * nv * tau / 2)) / U)
    ev, er = (float(np.sqrt(np.mean(np.square(e)))) for e in (ev, er))
    print(f"r 2^{log_r} m 2^{log_m} eps {eps:.1e}: {weak.mean():.2f} weak, dv {ev:.2f} dr {er:.2f}")
    assert ev <= bound_v and er <= bound_r
