"""Coefficients, kinematics and sectors at the edges of what the evaluators of
csrc/qmc_real.cuh and csrc/qmc_deformed.cuh take (GPU)."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads as w

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
