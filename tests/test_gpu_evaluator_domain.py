"""Coefficients, kinematics and sectors at the edges of what the evaluators of
csrc/qmc_real.cuh and csrc/qmc_deformed.cuh take (GPU)."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads as w
from paper_2305_19768_gb300.inputs.integral import Integral

from parity import Gpu
from test_gpu_real_integer import _compare, _specs, general

pytestmark = pytest.mark.gpu

NONFINITE = -7


class _Text:
    """Sector text for Gpu.load"""

    def __init__(self, text):
        self.text = text

    def to_text(self):
        return self.text


def _with_signed_zero(I):
    """Each U and F gets one more monomial t_1 .. t_d of coefficient -0.0; with
    +0.0 times negative invariants the coefficient stays -0.0 at the point."""
    out, d = [], 0
    for line in I.to_text().splitlines():
        tok = line.split()
        if tok[0] == "sector":
            d = int(tok[3])
        if tok[0] in ("U", "F") and len(tok) == 4:
            tok[3] = str(int(tok[3]) + 1)
            out.append(" ".join(tok))
            out.append(" ".join(["1"] * d + ["-0.0"] + ["0.0"] * len(I.invariants)))
        else:
            out.append(line)
    return _Text("\n".join(out) + "\n")


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("name", ["box", "double_box"])
def test_signed_zero_coefficients(name, mixed):
    """A coefficient of -0.0 changes nothing: the sums with and without it are
    two FP64 evaluations of one formula (the bar of test_gpu_real_integer)."""
    build, lo, kin = {"box": (w.box_massless, -2, [[-3.0, -2.0]]),
                      "double_box": (w.double_box_massless, -4, [[-3.0, -1.0]])}[name]
    I = build()
    g = Gpu(precision=qmc.QMC_PRECISION_MIXED if mixed else qmc.QMC_PRECISION_FP64)
    try:
        iid, zid = g.load(I), g.load(_with_signed_zero(I))
        qmc.qmc_set_kinematics(g.ctx, np.array(kin))
        specs = _specs(iid, I, name, 1, 1009, 2)
        nord = 1 - lo
        b, _, rb = g.eval(iid, specs, lo, nord)
        a, _, ra = g.eval(zid, [dict(sp, integral_id=zid) for sp in specs], lo, nord)
        assert ra == 0 and rb == 0
        _compare(I, specs, a, b, kin, 2, lo, nord, 0)
    finally:
        g.close()


@pytest.mark.parametrize("scale", [1e40, 1e22, 1e-22, 1e-42])
@pytest.mark.parametrize("name", ["box", "double_box"])
def test_mixed_coefficients_near_and_beyond_the_fp32_range(name, scale):
    """Where FP32 coefficients overflow or lose bits, mixed jobs give what the
    general kernel gives: its sums, or its status for sums that are not finite."""
    build, lo = (w.box_massless, -2) if name == "box" else (w.double_box_massless, -4)
    I = build()
    g = Gpu(precision=qmc.QMC_PRECISION_MIXED)
    try:
        iid, gid = g.load(I), g.load(general(I, Fraction(-1, 10 ** 250)))
        qmc.qmc_set_kinematics(g.ctx, np.array([[-3.0 * scale, -2.0 * scale]]))
        specs = _specs(iid, I, name, 1, 1009, 2)
        nord = 1 - lo
        a, _, ra = g.eval(iid, specs, lo, nord)
        b, _, rb = g.eval(gid, [dict(sp, integral_id=gid) for sp in specs], lo, nord)
        assert ra == rb
        if scale == 1e40 and name == "box":
            assert rb == NONFINITE
        if rb == 0:
            assert np.all(np.abs(a - b) <= 1e-9 * np.abs(b).max())
    finally:
        g.close()

TOY = """qmc-sectors 1
name toy
loops 1 propagators 3 dim 4
invariants 1 s
prefactor 0 1 1.0 0.0
nsectors 1
sector 0 d 1 deform 1
a 0
b 0.0
U 0.0 0.0 1
0 1.0 0.0
F {f0} {f1} 2
0 0.0 1.0
1 0.0 -2.0
end
"""


def _status(I, lo, nord, kin, lam, mixed=False, n=1009, z=None, transform=0, flags=0):
    """(general kernel's status, the job's own)"""
    g = Gpu(transform=transform, precision=qmc.QMC_PRECISION_MIXED if mixed else qmc.QMC_PRECISION_FP64)
    try:
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array([kin]))
        J = Integral.from_text(I.to_text())
        specs = [dict(integral_id=iid, sector=s, point=0, shifts=1 if flags else 2, n=n, seed=3, stream=s, flags=flags,
                      **{"lambda": lam}, **({} if z is None else {"z": z})) for s in range(len(J.sectors))]
        got = g.eval(iid, specs, lo, nord)[2]
        gid = g.load(general(J, Fraction(1, 10 ** 250)))
        return g.eval(gid, [dict(sp, integral_id=gid) for sp in specs], lo, nord)[2], got
    finally:
        g.close()


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("s", [0.0, 1e160, 1e-170])
@pytest.mark.parametrize("name,lo,nord", [("triangle", -2, 3), ("bubble", -1, 3)])
def test_zero_and_unrepresentable_F_are_reported(name, lo, nord, s, mixed):
    """F = 0 everywhere (s = 0), also where only its logarithm enters (the bubble
    to eps^1), and |F|^2 outside FP64's normal range: the sums are not finite,
    and the status says so, as with the general kernel."""
    I = w.triangle_one_offshell(0, "s") if name == "triangle" else w.bubble(0, "s")
    ref, got = _status(I, lo, nord, [s], 0.5, mixed)
    assert got == NONFINITE
    if not mixed:
        assert ref == NONFINITE


@pytest.mark.parametrize("f0,f1,nord,status", [(-1.0, 0.0, 1, NONFINITE), (-2.0, -1.0, 1, NONFINITE),
                                               (0.0, -1.0, 2, NONFINITE), (1.0, 0.0, 1, 0), (1.0, 0.0, 2, 0)])
def test_one_point_with_F_zero(f0, f1, nord, status):
    """F = s (1 - 2 t), undeformed (lambda = 0), unshifted lattice of 1024 points
    without a transform: F = 0 at t = 1/2, an error for a negative power or a
    logarithm and a plain zero for a positive power."""
    ref, got = _status(_Text(TOY.format(f0=f0, f1=f1)), 0, nord, [3.0], 0.0, n=1024, z=[1, 1, 1, 1, 1, 1],
                       transform=2, flags=qmc.QMC_JOB_UNSHIFTED)
    assert got == status and ref == status


@pytest.mark.parametrize("s", [9e-39, 9e-40, 9e-42, 9.0])
def test_mixed_deformed_keeps_fp32_subnormals(s):
    """F, its derivatives and the contour in FP32's subnormal range: the same
    FP32 values as in the general kernel, which serves a window up to eps^2."""
    I = w.bubble(0, "s")
    g = Gpu(precision=qmc.QMC_PRECISION_MIXED)
    try:
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array([[s]]))
        specs = [dict(integral_id=iid, sector=i, point=0, shifts=2, n=1009, seed=3, stream=i, **{"lambda": 0.5 / s})
                 for i in range(len(I.sectors))]
        a, fa, ra = g.eval(iid, specs, -1, 3)
        b, fb, rb = g.eval(iid, specs, -1, 4)
        assert ra == rb == 0 and fa == fb
        a, b = a.reshape(-1, 3, 2), b.reshape(-1, 4, 2)[:, :3]
        assert np.all(np.abs(a - b) <= 1e-11 * np.abs(b).max())
    finally:
        g.close()


@pytest.mark.parametrize("lam", [1e-3, 1e-6, 1e-9])
def test_imaginary_parts_of_nearly_real_sums(lam):
    """With a small lambda at Euclidean kinematics every argument is small and
    the sums' imaginary parts are proportional to it: the same relative accuracy
    as the general kernel's. Six points a sum, so that neither the corners nor the
    points cancel by more than 10^3: some 10^3 2^-53 each side, bar 1e-11."""
    I, lo, kin = w.box_massless(deform=True), -2, [-3.0, -2.0]
    g = Gpu()
    try:
        iid, gid = g.load(I), g.load(general(I, Fraction(1, 10 ** 250)))
        qmc.qmc_set_kinematics(g.ctx, np.array([kin]))
        specs = [dict(integral_id=iid, sector=s, point=0, shifts=1, n=7, z=[1, 2, 3, 1, 1, 1], seed=3, stream=s,
                      flags=qmc.QMC_JOB_UNSHIFTED, **{"lambda": lam}) for s in range(len(I.sectors))]
        for hi in (0, 1):
            nord = hi - lo + 1
            a, _, ra = g.eval(iid, specs, lo, nord)
            b, _, rb = g.eval(gid, [dict(sp, integral_id=gid) for sp in specs], lo, nord)
            assert ra == rb == 0
            a, b = a.reshape(-1, nord, 2)[..., 1], b.reshape(-1, nord, 2)[..., 1]
            top = np.abs(b).max(axis=0)
            assert top[-1] > 0 and np.all(np.abs(a - b) <= 1e-11 * top), np.abs(a - b).max(axis=0) / top
    finally:
        g.close()


FAR = """qmc-sectors 1
name far
loops 2 propagators 7 dim 4
invariants 1 s
prefactor 0 1 1.0 0.0
nsectors 1
sector 0 d 6 deform 0
a -1 4 -1 4 -1 4
b -1.0 0.0 -2.0 0.0 1.0 0.0
U 1.0 3.0 2
0 0 0 0 0 0 1.0 0.0
1 1 1 0 0 0 1.0 0.0
F -2.0 -2.0 3
0 0 0 0 0 0 0.0 -1.0
1 0 0 1 1 0 0.0 -1.0
0 1 1 0 0 1 1.0 0.0
end
"""


def test_prefactors_below_the_normal_range():
    """Regular factors t^4 in three variables at the first points of an unshifted
    lattice with n = 2^24 (t = 35 / n^4 each): their product is below FP64's normal
    range, and the sums are the general kernel's."""
    g = Gpu()
    try:
        J = Integral.from_text(FAR)
        iid, gid = g.load(J), g.load(general(J, Fraction(-1, 10 ** 250)))
        qmc.qmc_set_kinematics(g.ctx, np.array([[-3.0]]))
        sp = dict(integral_id=iid, sector=0, point=0, shifts=1, n=16777259, z=[1] * 6, seed=3, stream=0,
                  flags=qmc.QMC_JOB_UNSHIFTED)
        a, _, ra = g.eval(iid, [sp], -3, 4)
        b, _, rb = g.eval(gid, [dict(sp, integral_id=gid)], -3, 4)
        assert ra == rb == 0
        assert np.all(np.abs(a - b) <= 1e-11 * np.abs(b).max())
    finally:
        g.close()


@pytest.mark.parametrize("lam", [float("nan"), float("inf"), -float("inf"), 1e-250, -1e-290, 5e-324])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("name", ["box_massive", "box"])
def test_lambda_outside_the_usual_range(name, lam, mixed):
    """A lambda that is not finite gives sums that are not, and the status says
    so; one whose products leave FP64's normal range gives the undeformed sums."""
    I, lo = (w.box_massive(), 0) if name == "box_massive" else (w.box_massless(deform=True), -2)
    g = Gpu(precision=qmc.QMC_PRECISION_MIXED if mixed else qmc.QMC_PRECISION_FP64)
    try:
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array([[-3.0, -2.0]]))
        specs = [dict(integral_id=iid, sector=s, point=0, shifts=2, n=1009, seed=3, stream=s, **{"lambda": lam})
                 for s in range(len(I.sectors))]
        a, _, ra = g.eval(iid, specs, lo, 1 - lo)
        if not np.isfinite(lam):
            assert ra == NONFINITE
            return
        b, _, rb = g.eval(iid, [dict(sp, **{"lambda": 0.0}) for sp in specs], lo, 1 - lo)
        assert ra in (0, -6) and rb == 0            # (-6: a negative lambda's sign check)
        assert np.all(np.abs(a - b) <= 1e-12 * np.abs(b).max())
    finally:
        g.close()


@pytest.mark.parametrize("scale", [1e70, 1e75, 1e78, 1e90, 1e120, 1e-70, 1e-78])
def test_deformed_coefficients_of_any_size(scale):
    """F^-2 at large and small kinematics: the general kernel's sums where it has
    them, and its status where the square of F^2 leaves FP64's range."""
    I, lo = w.box_massless(deform=True), -2
    g = Gpu()
    try:
        iid, gid = g.load(I), g.load(general(I, Fraction(1, 10 ** 250)))
        qmc.qmc_set_kinematics(g.ctx, np.array([[7.0 * scale, -2.5 * scale]]))
        specs = [dict(integral_id=iid, sector=s, point=0, shifts=2, n=1009, seed=3, stream=s,
                      **{"lambda": 0.5 / scale}) for s in range(len(I.sectors))]
        a, fa, ra = g.eval(iid, specs, lo, 3)
        b, fb, rb = g.eval(gid, [dict(sp, integral_id=gid) for sp in specs], lo, 3)
        assert ra == rb and rb == (0 if 1e-76 < scale < 1e76 else NONFINITE)
        if rb == 0:
            a, b = a.reshape(-1, 3, 2), b.reshape(-1, 3, 2)
            top = np.abs(b).max(axis=(0, 2))
            assert np.all(top > 0) and np.all(np.abs(a - b).max(axis=(0, 2)) <= 1e-11 * top)
    finally:
        g.close()


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("s", [1e30, 1e60, 1e160])
def test_sign_failures_where_F_is_not_a_number(s, mixed):
    """Points whose F is NaN fail no sign check: the same counts as the general
    kernel's, which serves a window up to eps^2."""
    I = w.box_massive()
    g = Gpu(precision=qmc.QMC_PRECISION_MIXED if mixed else qmc.QMC_PRECISION_FP64)
    try:
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array([[s, -0.3 * s]]))
        specs = [dict(integral_id=iid, sector=i, point=0, shifts=2, n=1009, seed=3, stream=i, **{"lambda": 0.5})
                 for i in range(len(I.sectors))]
        _, fa, ra = g.eval(iid, specs, 0, 1)
        _, fb, rb = g.eval(iid, specs, 0, 3)
        assert fa == fb and (ra == rb or not mixed)
    finally:
        g.close()
