"""The integer arctangent of csrc/qmc_iarg.h, built with g++ on the CPU, against
50-digit arguments: relative error at every size of the argument, the quadrants,
the F - i0 prescription, and sums of multiples."""
import ctypes
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

from test_kernel_math_host import CSRC

mp = pytest.importorskip("mpmath")

HARNESS = r"""
#include <cstdint>
#include <cstring>
#include "qmc_iarg.h"
extern "C" void args(const double *y, const double *x, const int64_t *tab, int m0, uint64_t *m, int32_t *e,
                     int32_t *s, long n) {
    for (long i = 0; i < n; ++i) {
        const qmc_xf r = qmc_iarg(y[i], x[i], m0 != 0, tab);
        m[i] = r.m; e[i] = r.e; s[i] = r.neg;
    }
}
extern "C" void sums(const double *y, const double *x, const int64_t *tab, const int32_t *k, double *out, long n) {
    for (long i = 0; i < n; ++i) {
        qmc_u128 s = 0;
        for (int f = 0; f < 5; ++f) s = qmc_iarg_add(s, qmc_iarg(y[5 * i + f], x[5 * i + f], false, tab), k[5 * i + f]);
        out[i] = qmc_iarg_sum(s);
    }
}
"""


def _ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("iarg")
    (d / "h.cpp").write_text(HARNESS)
    so = d / "libiarg.so"
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "h.cpp"), "-o", str(so)],
                   check=True, capture_output=True)
    return ctypes.CDLL(str(so))


def _table():
    """atan(j / 64) 2^63 as the kernel forms it from its two-word table"""
    text = open(os.path.join(CSRC, "qmc_log_table.h")).read()
    body = text[text.index("QMC_ATAN_TABLE_INIT"):]
    v = [float.fromhex(t) for t in re.findall(r"-?0x[01]\.[0-9a-f]+p[-+]\d+", body)[:130]]
    return np.array([round(v[2 * j] * 2.0 ** 63) + round(v[2 * j + 1] * 2.0 ** 63) for j in range(65)], dtype=np.int64)


def _args(lib, y, x, m0=0):
    y, x = np.ascontiguousarray(y, dtype=np.float64), np.ascontiguousarray(x, dtype=np.float64)
    tab = _table()
    m, e, s = np.empty(y.size, np.uint64), np.empty(y.size, np.int32), np.empty(y.size, np.int32)
    lib.args(_ptr(y), _ptr(x), _ptr(tab), m0, _ptr(m), _ptr(e), _ptr(s), ctypes.c_long(y.size))
    return [mp.ldexp(mp.mpf(int(a)), int(b) - 63) * (-1 if c else 1) if a else mp.mpf(0) for a, b, c in zip(m, e, s)]


def test_relative_error_at_every_size(lib):
    mp.mp.dps = 50
    rng = np.random.default_rng(3)
    n = 3000
    x = rng.normal(size=n)
    y = np.concatenate([rng.normal(size=n), x * 2.0 ** rng.uniform(-900, 0, n), x * 2.0 ** rng.uniform(-12, 12, n)])
    x = np.concatenate([x, x, x])
    # ratios at the ends of the table's cells and of the cells' halves, mantissas near 2
    c = np.arange(1, 129) / 128.0
    big = 2.0 - 2.0 ** -52 * rng.integers(1, 9, 128 * 8)
    y = np.concatenate([y, np.repeat(c, 8) * big, [5e-324, 1e-310, 2.0, 1e-320, 1.0, 1.0]])
    x = np.concatenate([x, big, [1.0, 3e-308, 2.0, 1e300, 1e-320, -1e-320]])
    for sy, sx in ((1, 1), (1, -1), (-1, 1), (-1, -1)):
        for g, a, b in zip(_args(lib, sy * y, sx * x), sy * y, sx * x):
            ref = mp.atan2(mp.mpf(float(a)), mp.mpf(float(b)))
            assert abs(g - ref) <= abs(ref) * mp.mpf(2) ** -55, (a, b)


def test_zeros_and_the_prescription(lib):
    pi = float(mp.pi)
    for y, x, m0, ref in ((0.0, 2.0, 0, 0.0), (0.0, -2.0, 0, pi), (-0.0, -2.0, 0, -pi), (0.0, -2.0, 1, -pi),
                          (0.0, 2.0, 1, 0.0), (3.0, 0.0, 0, pi / 2), (-3.0, 0.0, 1, -pi / 2), (0.0, 0.0, 0, 0.0)):
        assert float(_args(lib, [y], [x], m0)[0]) == ref


def test_sums_of_five(lib):
    """Sums k_1 a_1 + .. + k_5 a_5, |k| <= 4, at their largest and with small
    arguments: half a unit of the result, and of every term 2^-55 and 4 2^-120."""
    mp.mp.dps = 50
    rng = np.random.default_rng(4)
    n = 1500
    x, y = rng.normal(size=(n, 5)), rng.normal(size=(n, 5))
    y[500:1000] *= 2.0 ** rng.uniform(-70, 0, (500, 1))
    y[1000:], x[1000:] = -1e-17, -1.0
    k = rng.integers(-4, 5, (n, 5)).astype(np.int32)
    k[1000:] = 4
    out, tab = np.empty(n), _table()
    lib.sums(_ptr(y), _ptr(x), _ptr(tab), _ptr(k), _ptr(out), ctypes.c_long(n))
    for a, b, f, g in zip(y, x, k, out):
        terms = [int(q) * mp.atan2(mp.mpf(float(v)), mp.mpf(float(u))) for v, u, q in zip(a, b, f)]
        ref = sum(terms)
        bar = abs(ref) * mp.mpf(2) ** -53 + sum(abs(t) for t in terms) * mp.mpf(2) ** -55 + 20 * mp.mpf(2) ** -120
        assert abs(mp.mpf(float(g)) - ref) <= bar
