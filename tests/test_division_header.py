"""The pivot search's division (csrc/division.cuh) itself, compiled for the host, against IEEE
division bit for bit: on both sides of the exponent bounds inside which it takes its own
steps, and for zeros, subnormals, infinities and NaN."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1305_2353_gb300", "csrc")
C = r"""
#include "division.cuh"
extern "C" void run(long n, const double *x, const double *d, double *q) {
    for (long i = 0; i < n; i++) q[i] = div_by(x[i], d[i], 1.0 / d[i]);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("div")
    (d / "div.cpp").write_text(C)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-I", CSRC, "-shared", "-fPIC", "-o", str(d / "div.so"),
                    str(d / "div.cpp"), "-lm"], check=True)
    L = ctypes.CDLL(str(d / "div.so"))
    L.run.argtypes = [ctypes.c_long] + [ctypes.c_void_p] * 3
    return L


def _same(lib, x, d):
    x, d = np.ascontiguousarray(x), np.ascontiguousarray(d)
    q = np.empty_like(x)
    lib.run(len(x), x.ctypes.data, d.ctypes.data, q.ctypes.data)
    with np.errstate(all="ignore"):
        want = x / d
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(q), nan)
    assert np.array_equal(q[~nan].view(np.uint64), want[~nan].view(np.uint64))


def _values(rng, exponents, n):
    m = np.where(rng.random(n) < 0.3, 2 ** 52 - 1 - rng.integers(0, 8, n), rng.integers(0, 2 ** 52, n)).astype(np.uint64)
    v = (m | (rng.choice(exponents, n).astype(np.uint64) << np.uint64(52))).view(np.float64)
    return np.where(rng.random(n) < 0.5, -v, v)


@pytest.mark.parametrize("ex", [range(396, 405), range(1000, 1050), range(1642, 1651), [0, 1, 2, 2046]])
@pytest.mark.parametrize("ed", [range(719, 728), range(1000, 1050), range(1319, 1328), [0, 1, 2, 2045, 2046]])
def test_both_sides_of_the_bounds(lib, ex, ed):
    rng = np.random.default_rng(len(ex) + len(ed))
    _same(lib, _values(rng, list(ex), 200_000), _values(rng, list(ed), 200_000))


def test_special_operands(lib):
    s = np.array([0.0, -0.0, 5e-324, -5e-324, 2.2e-308, 1.0, -1.0, 3.0, 1.7e308, np.inf, -np.inf, np.nan])
    _same(lib, np.repeat(s, len(s)), np.tile(s, len(s)))
