"""The polynomial of the integer logarithm (csrc/qmc_ilog.h) on the CPU: its
results against the same reduction with the polynomial in exact arithmetic.
Its roundings (below 2^-73 of log1p, and 2^-116) change none of some 36000."""
import numpy as np

from test_kernel_math_host import CSRC, ilog  # noqa: F401  (fixture)


def _table():
    import os
    import re

    text = open(os.path.join(CSRC, "qmc_log_table.h")).read()
    body = text[text.index("QMC_LOG_TABLE_INIT"):]
    return [int(x, 16) for x in re.findall(r"0x[0-9a-fA-F]+", body)[:3 * 1025]]


def _exact(x, tab):
    """RN of e ln 2 + ln F + f (1 - f (1/2 - f/3 + f^2/4 - f^3/5 + f^4/6)), the
    table's ln 2, ln F and f as the kernel has them and the polynomial exact"""
    m, e = np.frexp(x)
    e = int(e) - 1
    frac = int(m * 2.0 ** 64) - (1 << 63)
    j = (frac + (1 << 52)) >> 53
    r = frac - (j << 53)
    f = (abs(r) * tab[3 * j] >> 52) * (-1 if r < 0 else 1)              # f 2^74
    one = 1 << 74
    p, q = 0, 60                                                        # q p(f) by Horner, q = 60
    for k in (6, 5, 4, 3, 2):
        p = q // k * one ** (6 - k) - f * p                             # scaled 2^(74 (6 - k))
    lp = f * (q * one ** 5 - f * p)                                     # q 2^(74 * 6) log1p f
    lnf = (tab[3 * j + 2] << 64) | tab[3 * j + 1]
    ln2 = (0xb17217f7d1cf7 << 64) | 0x9abc9e3b39803f2f
    scale = 74 * 6 - 116
    S = (lnf + e * ln2) * q * (1 << scale) + lp                         # q 2^(74 * 6) ln x
    if S == 0:
        return 0.0
    a, den = abs(S), q << (74 * 6)
    sh = a.bit_length() - den.bit_length() - 53
    num, d = (a << -sh, den) if sh < 0 else (a, den << sh)
    n, rem = divmod(num, d)
    while n >= 1 << 53:
        num, d, sh = num, d << 1, sh + 1
        n, rem = divmod(num, d)
    n += 1 if (2 * rem > d or (2 * rem == d and n & 1)) else 0
    return float(np.ldexp(float(n), sh)) * (-1 if S < 0 else 1)


def test_polynomial_costs_no_result_its_rounding(ilog):  # noqa: F811
    rng = np.random.default_rng(23)
    k = np.arange(1, 2001, dtype=np.float64)
    F = 1.0 + np.arange(1025) / 1024.0
    x = np.concatenate([1.0 + k * 2.0 ** -52, 1.0 - k * 2.0 ** -53, 1.0 + rng.uniform(-2.0 ** -11, 2.0 ** -11, 20000),
                        ((F[:-1] + 0.5 / 1024)[:, None] * (1 + rng.uniform(-1e-9, 1e-9, (1024, 4)))).ravel(),
                        rng.uniform(0.5, 2.0, 4000), np.exp(rng.uniform(-700, 700, 4000))])
    got, tab = ilog(x), _table()
    ref = np.array([_exact(v, tab) for v in x])
    assert np.abs(got - ref).max() <= np.spacing(700.0)
    assert np.array_equal(got, ref), int((got != ref).sum())
