"""CPU check of the FP32 weak pair map (csrc/kepler_weak32.cuh), built as host
C++, against the Kepler map in double precision."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("weak32") / "libweak32.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                    os.path.join(HERE, "weak32_host.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


def _weak32(lib, x, v, m, tau, post):
    n = m.shape[0]
    weak, out = np.zeros(n, np.int32), np.zeros((n, 6), np.float32)
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (x, v, m, tau)]
    lib.weak32(ctypes.c_long(n), *p, ctypes.c_float(post),
               weak.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p))
    return weak.astype(bool), out.astype(np.float64)


def _exact(x, v, m, t, post):
    x, v, m, t = (np.asarray(a, np.float64) for a in (x, v, m, t))
    r0, eta, v2 = np.sqrt((x * x).sum(1)), (x * v).sum(1), (v * v).sum(1)
    beta = 2 * m / r0 - v2
    zeta = m - beta * r0

    def G(s):
        y, g = -beta * s * s, []
        for j in range(4):
            term, acc = 1.0 / (1, 1, 2, 6)[j], 0.0
            for k in range(12):
                acc, term = acc + term, term * y / ((2 * k + j + 1) * (2 * k + j + 2))
            g.append(acc * s ** j)
        return g
    s = t / r0
    for _ in range(8):
        g = G(s)
        s = s - (r0 * s + eta * g[2] + zeta * g[3] - t) / (r0 + eta * g[1] + zeta * g[2])
    g = G(s)
    r = r0 + eta * g[1] + zeta * g[2]
    fd, gd = -g[1] / (r0 * r), -g[2] / r
    A, B = -g[2] / r0 - post * t * fd, -g[3] - post * t * gd
    return np.concatenate([A[:, None] * x + B[:, None] * v, fd[:, None] * x + gd[:, None] * v], 1)


@pytest.mark.parametrize("post", [0.0, 0.5, 1.0])
@pytest.mark.parametrize("scale", [1e-6, 1.0, 1e9])
def test_increments_within_the_rounding_of_their_chain(lib, post, scale):
    # some 12 roundings of half a unit in a chain and 1.5 of the separation's
    # and its root's: at most 12 units of 2^-24 of the velocity increment, and
    # as much of |t delta_v| for the position's
    rng = np.random.default_rng(int(post * 2) + 3)
    n = 20000
    x = (rng.uniform(-1, 1, (n, 3)) * scale).astype(np.float32)
    v = rng.uniform(-1, 1, (n, 3)).astype(np.float32)
    r0 = np.linalg.norm(x.astype(np.float64), axis=1)
    eps = np.exp2(-rng.uniform(4.0, 16.0, n))
    tau = (rng.choice([-1, 1], n) * eps * r0 / np.linalg.norm(v, axis=1)).astype(np.float32)
    m = (np.exp2(-rng.uniform(8.0, 20.0, n)) * r0 ** 3 / tau.astype(np.float64) ** 2
         ).astype(np.float32)
    weak, out = _weak32(lib, x, v, m, tau, post)
    assert weak.mean() > 0.95
    ref = _exact(x, v, m, tau, post)
    dv = np.linalg.norm(ref[:, 3:], axis=1)
    ev = np.linalg.norm(out[:, 3:] - ref[:, 3:], axis=1) / dv
    er = np.linalg.norm(out[:, :3] - ref[:, :3], axis=1) / (dv * abs(tau))
    assert ev[weak].max() <= 12 * 2.0 ** -24 and er[weak].max() <= 12 * 2.0 ** -24


def test_pairs_beyond_the_limits_are_left_to_the_general_solve(lib):
    one = lambda a: np.array([a], np.float32)
    for x, v, m, t in (([1, 0, 0], [0.07, 0, 0], 1e-3, 1.0),       # |w| > 2^-4 r0
                       ([1, 0, 0], [0, 0, 0], 5e-3, 1.0),          # mu > 2^-8
                       ([0, 0, 0], [0, 0, 0], 1e-3, 1.0),          # coincident
                       ([1e25, 0, 0], [0, 0, 0], 1e-3, 1.0),       # r0^2 beyond float
                       ([1, 0, 0], [np.nan, 0, 0], 1e-3, 1.0),
                       ([1e-25, 0, 0], [0, 0, 0], 1e-18, 1e-35)):  # t / r0^3 beyond float
        with np.errstate(all="ignore"):
            weak, _ = _weak32(lib, np.array([x], np.float32), np.array([v], np.float32), one(m),
                              one(t), 0.5)
        assert not weak[0], (x, v, m, t)
    weak, out = _weak32(lib, np.array([[1, 2, 3]], np.float32), np.array([[3, 1, 2]], np.float32),
                        one(1e-3), one(0.0), 0.5)
    assert weak[0] and not out.any()
