"""CPU check that the weak pair map (csrc/kepler_weak.cuh) is no less accurate
than the map in plain 64-bit arithmetic, up to the limits of its class."""
import numpy as np
import pytest

mpmath = pytest.importorskip("mpmath")

from test_weak_host import _cases, _exact, _run, lib  # noqa: E402,F401


def _plain(ri, vi, rj, vj, m, tau):
    """The second-order pair map over m in float64: drift, difference, drift
    back, the universal Kepler equation and the increments (Eqs. 17, 26)."""
    dot = lambda a, b: (a * b).sum(1)
    v = vi - vj
    x = ((ri + 0.5 * tau * vi) - (rj + 0.5 * tau * vj)) - 0.5 * tau * v
    r0 = np.sqrt(dot(x, x))
    eta, beta = dot(x, v), 2.0 * m / r0 - dot(v, v)
    zeta = m - beta * r0

    def G(s):
        y = beta * s * s
        c2 = 0.5 - y / 24.0 * (1.0 - y / 30.0 * (1.0 - y / 56.0 * (1.0 - y / 90.0)))
        c3 = (1.0 - y / 20.0 * (1.0 - y / 42.0 * (1.0 - y / 72.0 * (1.0 - y / 110.0)))) / 6.0
        return s * (1.0 - y * c3), s * s * c2, s * s * s * c3
    s = tau / r0
    for _ in range(6):
        g1, g2, g3 = G(s)
        s = s - (r0 * s + eta * g2 + zeta * g3 - tau) / (r0 + eta * g1 + zeta * g2)
    g1, g2, g3 = G(s)
    r = r0 + eta * g1 + zeta * g2
    return -(g1 / (r0 * r))[:, None] * x - (g2 / r)[:, None] * v


@pytest.mark.parametrize("seed", [1, 2, 3])
@pytest.mark.parametrize("lo,hi", [(2.0 ** -12, 2.0 ** -9), (2.0 ** -7, 2.0 ** -6),
                                   (2.0 ** -6, 2.0 ** -5.5), (2.0 ** -5.5, 2.0 ** -5)])
def test_weak_map_is_as_accurate_as_plain_float64(lib, lo, hi, seed):  # noqa: F811
    ri, vi, mi, rj, vj, mj, tau = _cases(np.random.default_rng(seed), 400, lo, hi)
    weak, inc, rest = _run(lib, ri, vi, mi, rj, vj, mj, tau)
    assert weak.mean() > 0.8
    plain = _plain(ri, vi, rj, vj, mi + mj, tau)
    err = {"weak": [], "plain": []}
    with mpmath.workdps(40):
        f = mpmath.mpf
        for k in np.flatnonzero(weak):
            _, dv = _exact(ri[k], vi[k], rj[k], vj[k], f(mi[k]) + f(mj[k]), tau)
            nv = mpmath.sqrt(sum(q * q for q in dv))
            got = {"weak": [(f(inc[k, 3 + q]) + f(rest[k, 3 + q])) / f(mj[k]) for q in range(3)],
                   "plain": [f(plain[k, q]) for q in range(3)]}
            for name, g in got.items():
                err[name].append(float(sum((a - b) ** 2 for a, b in zip(g, dv)) / nv ** 2))
    w, p = (2.0 ** 53 * np.sqrt(np.mean(err[name])) for name in ("weak", "plain"))
    print(f"eps {lo:.1e}..{hi:.1e}: weak {w:.2f}, plain {p:.2f} units of 2^-53")
    assert w <= p
