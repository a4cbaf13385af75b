"""CPU check of the conversions between double and double-word that the strong
pairs' double-word solve uses (csrc/kepler_weak.cuh)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("strong") / "libstronghost.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", "-shared",
                    "-fPIC", os.path.join(HERE, "strong_host.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _split(lib, x):
    h, l = np.zeros(x.size, np.float32), np.zeros(x.size, np.float32)
    lib.strong_split(ctypes.c_long(x.size), _p(x), _p(h), _p(l))
    return h, l


def test_split_is_the_nearest_float_and_the_nearest_rest(lib):
    rng = np.random.default_rng(5)
    x = rng.choice([-1.0, 1.0], 60000) * rng.uniform(1, 2, 60000) * 2.0 ** rng.integers(-90, 120, 60000)
    # the ends of a binade and the ties between two floats
    edge = np.array([1.0, 2.0 - 2.0 ** -52, 2.0 - 2.0 ** -24, 2.0 - 2.0 ** -25, 1.0 + 2.0 ** -24,
                     1.0 + 2.0 ** -24 - 2.0 ** -52, 1.0 + 2.0 ** -52, 1.0 + 2.0 ** -23])
    x[:16] = np.concatenate([edge, -edge])
    h, l = _split(lib, x)
    tie = np.abs(x - h.astype(np.float64)) == np.spacing(np.abs(h)).astype(np.float64) / 2
    assert np.all((h == x.astype(np.float32)) | tie)
    assert np.all(np.abs(x - h.astype(np.float64)) <= 2.0 ** -24 * np.abs(x))
    assert np.array_equal(l, (x - h.astype(np.float64)).astype(np.float32))


def test_split_outside_of_floats_range(lib):
    x = np.array([0.0, -0.0, 5e-324, 1e-300, -1e-40, 1e40, -1e300, np.inf, -np.inf, np.nan])
    h, l = _split(lib, x)
    assert np.all(h[:5] == 0) and np.all(l[:5] == 0) and not np.any(np.isfinite(h[5:]))


def test_join_is_exact_to_the_sums_rounding(lib):
    rng = np.random.default_rng(6)
    h = (rng.choice([-1.0, 1.0], 30000) * 2.0 ** rng.uniform(-126, 127, 30000)).astype(np.float32)
    l = (h * rng.uniform(-2.0 ** -24, 2.0 ** -24, 30000)).astype(np.float32)
    l[:100], h[100:110], l[100:110] = 0.0, 0.0, 0.0
    out = np.zeros(h.size)
    lib.strong_join(ctypes.c_long(h.size), _p(h), _p(l), _p(out))
    assert np.array_equal(out, h.astype(np.float64) + l.astype(np.float64))
