"""CPU check of the weak pair map (csrc/kepler_weak.cuh), built as host C++:
its increments against the exact Kepler map at 40 digits, over the pairs the
class test admits, up to its limits and over many scales."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

mpmath = pytest.importorskip("mpmath")
HERE = os.path.dirname(os.path.abspath(__file__))
U = 2.0 ** -53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("weak") / "libweakhost.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", "-shared",
                    "-fPIC", os.path.join(HERE, "weak_host.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _run(lib, ri, vi, mi, rj, vj, mj, tau):
    n = mi.shape[0]
    weak = np.zeros(n, np.int32)
    inc = np.zeros((n, 12))
    rest = np.zeros((n, 12))
    a = [np.ascontiguousarray(q, dtype=np.float64) for q in (ri, vi, mi, rj, vj, mj)]
    lib.weak_pairs(ctypes.c_long(n), *[_p(q) for q in a], ctypes.c_double(tau), _p(weak), _p(inc),
                   _p(rest))
    return weak.astype(bool), inc, rest


def _exact(ri, vi, rj, vj, m, tau):
    """Increments over m of the second-order pair map (positions, velocities)
    and r0, in 40 digits: series in the universal variable, Newton steps."""
    with mpmath.workdps(40):
        f = mpmath.mpf
        x = [f(float(a)) - f(float(b)) for a, b in zip(ri, rj)]
        v = [f(float(a)) - f(float(b)) for a, b in zip(vi, vj)]
        t = f(tau)
        dot = lambda a, b: sum(p * q for p, q in zip(a, b))
        r0 = mpmath.sqrt(dot(x, x))
        eta, v2 = dot(x, v), dot(v, v)
        beta = 2 * m / r0 - v2
        zeta = m - beta * r0

        def G(s):
            y = beta * s * s
            c = [sum((-y) ** k / mpmath.factorial(2 * k + j) for k in range(12)) for j in range(4)]
            return [c[j] * s ** j for j in range(4)]
        s = t / r0
        for _ in range(8):
            g = G(s)
            s -= (r0 * s + eta * g[2] + zeta * g[3] - t) / (r0 + eta * g[1] + zeta * g[2])
        g = G(s)
        r = r0 + eta * g[1] + zeta * g[2]
        fd, gd = -g[1] / (r0 * r), -g[2] / r
        A, B = -g[2] / r0 - t / 2 * fd, -g[3] - t / 2 * gd
        return ([A * a + B * b for a, b in zip(x, v)], [fd * a + gd * b for a, b in zip(x, v)])


def _cases(rng, n, eps_lo, eps_hi, log_r=0.0):
    """n pairs at separation 2^log_r, moving by a part of it between eps_lo
    and eps_hi, mu up to 2^-10, at a step of 2^-8; the pair's centre moves
    too."""
    unit = lambda: (lambda a: a / np.linalg.norm(a, axis=1)[:, None])(rng.normal(size=(n, 3)))
    tau, r0 = 2.0 ** -8, 2.0 ** log_r * np.exp(rng.uniform(-0.3, 0.3, n))
    x = unit() * r0[:, None]
    w = unit() * (r0 * np.exp(rng.uniform(np.log(eps_lo), np.log(eps_hi), n)))[:, None]
    mu = 2.0 ** -rng.uniform(10.0, 30.0, n)
    m = mu * r0 ** 3 / tau ** 2
    part = rng.uniform(0.001, 0.999, n)
    c, vc = rng.normal(size=(n, 3)) * r0[:, None], 0.3 * w[::-1] / tau
    f = (1 - part)[:, None]
    return (c + f * x, vc + f * w / tau, part * m, c - (1 - f) * x, vc - (1 - f) * w / tau,
            (1 - part) * m, tau)


@pytest.mark.parametrize("lo,hi,bound_v,bound_r", [
    # r.m.s. bounds in units of 2^-53: the leading term's FP64 operations (r0^2,
    # its reciprocal root, the products with the mass and x) make 1.5; a
    # double-word's 2^-47 of a correction eps makes 64 eps, twice over for the
    # velocity; the position increment has no leading term
    (2.0 ** -20, 2.0 ** -12, 2.0, 0.5), (2.0 ** -9, 2.0 ** -8, 2.5, 1.0),
    (2.0 ** -6, 2.0 ** -5, 6.0, 4.0)])
@pytest.mark.parametrize("log_r", [-20.0, 0.0, 20.0])
def test_weak_map_against_the_exact_one(lib, lo, hi, bound_v, bound_r, log_r):
    rng = np.random.default_rng(100 + int(-np.log2(hi)) + int(log_r))
    ri, vi, mi, rj, vj, mj, tau = _cases(rng, 300, lo, hi, log_r)
    weak, inc, rest = _run(lib, ri, vi, mi, rj, vj, mj, tau)
    assert weak.sum() > 200
    ev, er = [], []
    for k in np.flatnonzero(weak):
        with mpmath.workdps(40):
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
    print(f"eps {lo:.1e}..{hi:.1e} r 2^{log_r:.0f}: dv {ev:.2f} u, dr {er:.2f} u")
    assert ev <= bound_v and er <= bound_r


def test_only_weak_finite_pairs_in_range_are_admitted(lib):
    rng = np.random.default_rng(3)
    ri, vi, mi, rj, vj, mj, tau = _cases(rng, 64, 2.0 ** -9, 2.0 ** -7)
    weak, _, _ = _run(lib, ri, vi, mi, rj, vj, mj, tau)
    assert weak.all()

    def none(**change):
        a = dict(ri=ri, vi=vi, mi=mi, rj=rj, vj=vj, mj=mj, tau=tau)
        a.update(change)
        return not _run(lib, **a)[0].any()
    big = rj.copy()
    big[:, 0] = np.inf
    assert none(rj=big) and none(rj=ri) and none(ri=ri * np.nan) and none(vj=vj * np.nan)
    assert none(ri=ri * 1e150) and none(ri=rj + (ri - rj) * 2.0 ** -40)
    assert none(vi=vj + (vi - vj) * 64) and none(vi=vi + 64.0, vj=vj + 64.0)
    assert none(mi=mi * 2 ** 32) and none(mi=-mi) and none(mj=mj * 0) and none(mi=mi * 1e-60)
    assert none(mi=mi * np.nan)


def test_exact_coordinates_and_squares(lib):
    rng = np.random.default_rng(1)
    y = (rng.uniform(1, 2, 4000) * 2.0 ** rng.integers(-40, 40, 4000)).astype(np.float32)
    y[:4] = [1.0, 2.0 ** 24 - 1, 1.4142135, 1.4142137]
    out = np.zeros(4000)
    lib.weak_squares(ctypes.c_long(4000), _p(y), _p(out))
    np.testing.assert_array_equal(out, y.astype(np.float64) ** 2)
    x = rng.normal(size=4000) * 2.0 ** rng.integers(-60, 30, 4000)
    x[:6] = [0.0, -0.0, 1.0, 2.0 - 2.0 ** -52, -1.0 - 2.0 ** -24, 1.0 + 2.0 ** -52]
    lib.weak_splits(ctypes.c_long(4000), _p(x), _p(out))
    assert np.all(np.abs(out - x) <= 2.0 ** -47 * np.abs(x)) and np.all(out[:2] == 0)
    z = np.array([1e-40, -1e-300, 5e-324])
    lib.weak_splits(ctypes.c_long(3), _p(z), _p(out))
    assert np.all(out[:3] == 0)


def test_integer_product_is_the_rounded_one(lib):
    rng = np.random.default_rng(2)
    a = rng.choice([-1.0, 1.0], 40000) * rng.uniform(1, 2, 40000) * 2.0 ** rng.integers(-300, 300, 40000)
    b = rng.choice([-1.0, 1.0], 40000) * rng.uniform(1, 2, 40000) * 2.0 ** rng.integers(-300, 300, 40000)
    edge = np.array([1.0, 1.0 + 2.0 ** -52, 1.5, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -26])
    a[:25], b[:25] = np.repeat(edge, 5), np.tile(edge, 5)
    out = np.zeros(40000)
    lib.weak_products(ctypes.c_long(40000), _p(a), _p(b), _p(out))
    # equal but for exact ties, which go up here and to even there
    off = out != a * b
    assert off.sum() <= 25 and np.all(np.abs(out - a * b) <= 2.0 ** -52 * np.abs(a * b))
