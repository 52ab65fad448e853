"""The pivot search's division by a known reciprocal (two steps of Markstein's
division, csrc/pivot_tests.cuh) against IEEE division, bit for bit: random
significands, ones near the ends of a binade and near-ties, both signs, and the
exponents up to the bounds inside which the kernels use it."""
import ctypes
import subprocess

import numpy as np
import pytest

C = r"""
#include <math.h>
#include <stdint.h>
long div_steps(long n, const double *x, const double *d, double *q) {
    long bad = 0;
    for (long i = 0; i < n; i++) {
        const double y = 1.0 / d[i];
        const double q0 = x[i] * y;
        const double q1 = fma(fma(-q0, d[i], x[i]), y, q0);
        const double q2 = fma(fma(-q1, d[i], x[i]), y, q1);
        q[i] = x[i] == 0.0 ? q0 : q2;
        const double w = x[i] / d[i];
        bad += !(q[i] == w && signbit(q[i]) == signbit(w));
    }
    return bad;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("div")
    (d / "div.c").write_text(C)
    subprocess.run(["gcc", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", str(d / "div.so"), str(d / "div.c"),
                    "-lm"], check=True)
    L = ctypes.CDLL(str(d / "div.so"))
    L.div_steps.restype = ctypes.c_long
    L.div_steps.argtypes = [ctypes.c_long] + [ctypes.c_void_p] * 3
    return L


def _significands(rng, n, how):
    if how == "random":
        return rng.integers(0, 2 ** 52, n, dtype=np.uint64)
    if how == "ends":  # the first and last few of a binade, all ones among them
        return np.where(rng.random(n) < 0.5, rng.integers(0, 64, n), 2 ** 52 - 1 - rng.integers(0, 64, n)).astype(np.uint64)
    return (rng.integers(0, 2 ** 26, n) * 2 ** 26).astype(np.uint64)  # short ones: exact quotients and ties


@pytest.mark.parametrize("hx", ["random", "ends", "short"])
@pytest.mark.parametrize("hd", ["random", "ends", "short"])
def test_division_steps(lib, hx, hd):
    rng = np.random.default_rng(len(hx) * 16 + len(hd))
    n = 1_000_000
    for ex, ed in (((1000, 1050), (1000, 1050)), ((400, 1647), (723, 1324))):
        x = (_significands(rng, n, hx) | (rng.integers(*ex, n).astype(np.uint64) << np.uint64(52))).view(np.float64)
        d = (_significands(rng, n, hd) | (rng.integers(*ed, n).astype(np.uint64) << np.uint64(52))).view(np.float64)
        x = np.where(rng.random(n) < 0.5, -x, x)
        d = np.where(rng.random(n) < 0.5, -d, d)
        x[:: 1000] = 0.0
        x[1:: 1000] = -0.0
        # quotients whose product with the divisor rounds back to the dividend: near-exact cases
        x[2:: 7] = (d * rng.integers(1, 1 << 30, n))[2:: 7]
        ok = (np.abs(x) < 2.0 ** 623) & ((x == 0) | (np.abs(x) > 2.0 ** -623))
        x, d = np.ascontiguousarray(x[ok]), np.ascontiguousarray(d[ok])
        q = np.empty_like(x)
        assert lib.div_steps(len(x), x.ctypes.data, d.ctypes.data, q.ctypes.data) == 0
