"""CPU check of the product on the integer pipe (csrc/kepler_weak.cuh): the
IEEE one, exact ties to even included."""
import ctypes

import numpy as np

from test_weak_host import _p, lib  # noqa: F401


def test_integer_product_is_the_ieee_one(lib):  # noqa: F811
    rng = np.random.default_rng(9)
    n = 200000
    # short significands, whose products with long ones end in ties often
    short = rng.integers(1, 64, n).astype(np.float64)
    full = rng.uniform(1, 2, n)
    a = np.where(rng.random(n) < 0.5, short, full) * 2.0 ** rng.integers(-300, 300, n)
    b = rng.choice([-1.0, 1.0], n) * rng.uniform(1, 2, n) * 2.0 ** rng.integers(-300, 300, n)
    edge = np.array([1.0, 1.0 + 2.0 ** -52, 1.5, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -26, 3.0, 1.25])
    a[:49], b[:49] = np.repeat(edge, 7), np.tile(edge, 7)
    out = np.zeros(n)
    lib.weak_products(ctypes.c_long(n), _p(a), _p(b), _p(out))
    assert np.array_equal(out, a * b)
