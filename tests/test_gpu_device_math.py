"""The library's own elementary functions, value by value, against correctly rounded ones."""
import ctypes as C
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def _apply(name, x):
    lib = C.CDLL(os.path.join(HERE, "cuda", "libmath_probe.so"))
    x = np.ascontiguousarray(x)
    y = np.empty_like(x)
    assert getattr(lib, name)(x.ctypes.data_as(C.c_void_p), y.ctypes.data_as(C.c_void_p), C.c_int(x.size)) == 0
    return y


def test_exponential_of_the_thermodynamics():
    """x in [-708, 0] densely, around the borders of its table (multiples of ln 2 / 64), tiny and denormal, and both
    sides of the cut at -708: less than two units in the last place, as the sum of what its steps lose."""
    assert np.finfo(np.longdouble).nmant >= 63
    rng = np.random.default_rng(1)
    edges = -np.arange(0, 65000) * (np.log(2) / 64)
    x = np.concatenate([-rng.uniform(0, 708, 400000), -rng.uniform(0, 1, 200000), -np.exp(rng.uniform(-90, 0, 100000)),
                        edges, np.nextafter(edges, 0), np.nextafter(edges, -1000),
                        [0.0, -0.0, -5e-324, -1e-310, -2.0 ** -54, -2.0 ** -53, -0.25, np.nextafter(-0.25, 0),
                         np.nextafter(-708.0, 0)]])
    x = x[x > -708.0]
    y = _apply("probe_exp", x)
    exact = np.exp(x.astype(np.longdouble))
    unit = np.spacing(np.nextafter(exact.astype(np.float64), 0)).astype(np.longdouble)   # of the binade below a power of two
    err = np.abs((y.astype(np.longdouble) - exact) / unit)
    assert err.max() < 2.0, (x[err.argmax()], err.max())
    far = _apply("probe_exp", np.array([-708.0, np.nextafter(-708.0, -1000), -1e4, -1e308, -np.inf]))
    assert np.array_equal(far, np.zeros(5))
    assert np.isnan(_apply("probe_exp", np.array([np.nan]))).all()


def test_reciprocal_of_the_network():
    """1 / d for d in [1, 2^126], all exponents and the values that sigmoids see, within one unit in the last place; 0
    beyond, where 1 / d is no normal number any more."""
    rng = np.random.default_rng(2)
    powers = 2.0 ** np.arange(0, 127)
    d = np.concatenate([powers, np.exp2(rng.uniform(0, 126, 500000)), 1 + np.exp(rng.uniform(-20, 87, 500000)),
                        1 + np.arange(1 << 16) * 2.0 ** -23]).astype(np.float32)
    d = np.unique(np.concatenate([d, np.nextafter(d, np.float32(0))]))
    d = d[(d >= 1) & (d <= np.float32(2.0 ** 126))]
    r = _apply("probe_reciprocal", d).astype(np.float64)
    exact = 1.0 / d.astype(np.float64)
    unit = np.spacing(np.nextafter(exact.astype(np.float32), np.float32(0))).astype(np.float64)
    err = np.abs(r - exact) / unit
    assert err.max() <= 1.0, (d[err.argmax()], err.max())
    beyond = np.array([np.nextafter(np.float32(2.0 ** 126), np.float32(3e38)), 1.5e38, 1 + np.exp(88.0)], dtype=np.float32)
    assert np.array_equal(_apply("probe_reciprocal", beyond), np.zeros(3, dtype=np.float32))
