"""The arithmetic of the FP64 basis kernels (musr_kernels_f64.cuh) element by element, in a small library
built beside the tests (f64_arith.cu), against numpy's long double: the logarithm over its octave, at
every edge of its table, next to 1 and outside the table's range; the reciprocals over and outside
theirs.  Bounds: the logarithm next to 1 2^-53 |ln x| + 2^-57 as stated at the function, elsewhere three
roundings (series, table entry, their sum); the reciprocal its last rounding."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib():
    from paper_1509_07685_gb300 import build
    src, out = os.path.join(HERE, "f64_arith.cu"), os.path.join(HERE, "_f64_arith.so")
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", out, src], check=True,
                   capture_output=True, text=True)
    dll = ctypes.CDLL(out)
    d = ctypes.c_double
    dll.f64_elementwise.argtypes = [ctypes.c_int, ctypes.POINTER(d), ctypes.POINTER(d), ctypes.c_int]
    dll.f64_factors.argtypes = [ctypes.c_int, d, d, d, d, d, d, ctypes.c_int, ctypes.POINTER(d)]
    return dll


def _ptr(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


def _map(lib, what, x):
    x = np.ascontiguousarray(x, dtype=np.float64)
    y = np.empty_like(x)
    assert lib.f64_elementwise(what, _ptr(x), _ptr(y), x.size) == 0
    return y


def _words(hi):
    return (np.asarray(hi, np.int64) << 32).view(np.float64)


def _around(x, k=3):
    """x and its k neighbours on either side."""
    bits = np.asarray(x).view(np.int64)
    return np.concatenate([bits + j for j in range(-k, k + 1)]).view(np.float64)


def _ln_error(lib, x):
    exact = np.log(x.astype(np.longdouble))
    return np.abs(_map(lib, 0, x) - exact).astype(np.float64), np.abs(exact).astype(np.float64)


def test_logarithm_next_to_one(lib):
    rng = np.random.default_rng(1)
    h = 2.0 ** -7
    edges = _words(np.arange(0x3FEFC000, 0x3FF02000, 0x200))
    x = np.concatenate([1.0 + h * rng.uniform(-1, 1, 400000), 1.0 + 2.0 ** -11 * rng.uniform(-1, 1.0, 200000),
                        1.0 + np.outer([-1, 1], 2.0 ** -np.arange(8.0, 53.0)).ravel(), _around(edges), [1.0]])
    err, size = _ln_error(lib, x)
    assert np.max(err / (2.0 ** -53 * size + 2.0 ** -57)) <= 1.0
    assert _map(lib, 0, [1.0])[0] == 0.0


def test_logarithm(lib):
    rng = np.random.default_rng(2)
    edges = _words(np.arange(0x3FE60000, 0x3FF80000, 0x200))
    x = np.concatenate([rng.uniform(0.5, 2.0, 300000), _around(edges), 2.0 ** rng.uniform(-1074, 1024, 300000),
                        _around(_words([0x01700000, 0x7E700000])), [5e-324, 2.0 ** -1022, 1.7976931348623157e308]])
    err, size = _ln_error(lib, x)
    assert np.max(err / (3.0 * 2.0 ** -53 * size + 2.0 ** -57)) <= 1.0


def test_reciprocals(lib):
    rng = np.random.default_rng(3)
    edges = _around(_words([0x00100000, 0x3FF00000, 0x7FD00000]))
    x = np.concatenate([2.0 ** rng.uniform(-1022, 1024, 300000), rng.uniform(1.0, 2.0, 300000), edges])
    exact = 1.0 / x.astype(np.longdouble)
    # half a unit in the last place (an absolute 2^-1075 where the result is subnormal), with 2^-60 of slack
    bound = 2.0 ** -53 * (1 + 2.0 ** -6) * exact + np.longdouble(2.0) ** -1075
    assert np.all(np.abs(_map(lib, 1, x) - exact) <= bound)
    exact = 1.0 / np.maximum(x, 1.0).astype(np.longdouble)
    bound = 2.0 ** -53 * (1 + 2.0 ** -6) * exact + np.longdouble(2.0) ** -1075
    assert np.all(np.abs(_map(lib, 2, x) - exact) <= bound)
    assert np.array_equal(_map(lib, 2, [0.0, -3.0, 0.25, 1.0]), np.ones(4))


PLAIN, TF, KT = 1, 2, 3  # musr_dev.h


@pytest.mark.parametrize("kind,sigma,kt", [(PLAIN, 0.05, 0.0), (TF, 0.05, 0.0), (KT, 0.0, 0.05)])
def test_gaussian_factors_do_not_drift_from_a_fresh_bin(lib, kind, sigma, kt):
    """The factor at a bin is the fresh bin's, times one rounding per step made since (31 at most, 15.5 on
    average), times a table entry: with the handful of roundings of these two the root mean square over
    all bins is that of a walk of 20 roundings, each uniform within 2^-53.  A step factor that is itself
    rounded to a double would add its error once per step, all with one sign."""
    iters, dt, nu = 128, 12.8 / 32768, 3.1
    P = np.zeros((iters * 256, 2))
    assert lib.f64_factors(kind, 0.0, sigma, kt, nu, dt, 0.0, iters, _ptr(P)) == 0
    t = np.arange(iters * 256) * np.longdouble(dt)
    if kind == KT:
        u = (np.longdouble(kt) * t) ** 2
        exact = (1 + 2 * (1 - u) * np.exp(-u / 2)) / 3
        got = P[:, 0].astype(np.longdouble)
    else:
        exact = np.exp(-(np.longdouble(sigma) * t) ** 2 / 2)
        got = np.hypot(P[:, 0].astype(np.longdouble), P[:, 1].astype(np.longdouble))
    err = ((got - exact) / exact).astype(np.float64)
    assert np.sqrt(np.mean(err ** 2)) <= np.sqrt(20.0 / 3.0) * 2.0 ** -53
