"""The two reciprocals of qmc_xf.h on the CPU: qmc_xf_rcp bit for bit against
its formula in Python's integers, qmc_xf_rcp3 against its error bound."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_19768_gb300", "csrc")

SRC = r"""
#include <cstdint>
#include <cstring>
#include "qmc_xf.h"
extern "C" void rcp(const uint64_t *a, uint64_t *m, int32_t *e, int third, long n) {
    for (long i = 0; i < n; ++i) {
        const qmc_xf r = third ? qmc_xf_rcp3(qmc_xf{a[i], 0, 0}) : qmc_xf_rcp(qmc_xf{a[i], 0, 0});
        m[i] = r.m;
        e[i] = r.e;
    }
}
"""


@pytest.fixture(scope="module")
def rcp(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rcp")
    (d / "rcp.cpp").write_text(SRC)
    so = d / "rcp.so"
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "rcp.cpp"), "-o", str(so)],
                   check=True)
    lib = ctypes.CDLL(str(so))

    def run(a, third):
        a = np.ascontiguousarray(a, np.uint64)
        m, e = np.zeros(a.size, np.uint64), np.zeros(a.size, np.int32)
        lib.rcp(*(ctypes.c_void_p(x.ctypes.data) for x in (a, m, e)), ctypes.c_int(third), ctypes.c_long(a.size))
        return m, e
    return run


def _mantissas():
    """Uniform ones, ones just above 1 (the FP32 seed at 2) and just below 2,
    the ends of the 24-bit seed's cells."""
    rng = np.random.default_rng(7)
    top = 1 << 63
    u = [int(x) | top for x in rng.integers(0, 1 << 63, 3000, dtype=np.uint64)]
    near = [top + k for k in (1, 2, 3)] + [top + (1 << k) + o for k in range(2, 63) for o in (-1, 0, 1)]
    far = [(1 << 64) - (1 << k) + o for k in range(1, 62) for o in (-1, 0, 1)]
    cell = [((int(x) | (1 << 23)) << 40) + o for x in rng.integers(0, 1 << 23, 500) for o in (0, (1 << 40) - 1)]
    return np.array([x for x in u + near + far + cell if x != top], dtype=object)


def _two_steps(m):
    """y <- y + y (1 - m y), twice, every product rounded down to Q62, from the
    FP32 reciprocal of the top 24 bits"""
    y0 = np.float32(1) / np.float32((m >> 40) / 2.0 ** 24)
    y = (1 << 63) - 1 if y0 >= 2 else int(float(y0) * 2 ** 62)
    for _ in range(2):
        e = (1 << 62) - (m * y >> 64)
        y += (y * e >> 64) << 2
    return y << 1


def test_two_step_reciprocal_is_its_formula(rcp):
    a = _mantissas()
    m, e = rcp(a.astype(np.uint64), 0)
    assert np.all(e == -1)
    assert [int(x) for x in m] == [_two_steps(int(x)) for x in a]


def test_third_order_reciprocal_within_2_61(rcp):
    """A value a 2^-63 of [1, 2) gives m 2^(e - 63)."""
    a = _mantissas()
    m, e = rcp(a.astype(np.uint64), 1)
    assert np.all(m >> np.uint64(63) == 1)
    for x, y, k in zip(a, m, e):
        assert abs(Fraction(int(x), 1 << 63) * Fraction(int(y), 1 << 63) * Fraction(2) ** int(k) - 1) < Fraction(1, 1 << 61)


def test_powers_of_two_are_exact(rcp):
    for third in (0, 1):
        m, e = rcp(np.array([1 << 63], dtype=np.uint64), third)
        assert int(m[0]) == 1 << 63 and int(e[0]) == 0
