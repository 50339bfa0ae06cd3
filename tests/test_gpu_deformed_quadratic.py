"""The deformed evaluator for quadratic F (csrc/qmc_deformed.cuh, GPU) against
the general deformed kernel, which takes F of higher degree, on everything it
accepts: one to three variables, zero to two of them singular, FP64 and (sums
to eps^1 against sums to eps^0) mixed precision, every transform; and
sectors it does not accept (F of higher degree), which stay on the general
kernel and still match the oracle."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads as w
from paper_2305_19768_gb300.inputs.integral import Integral
from paper_2305_19768_gb300.inputs.lattice import lattice_for

from parity import Gpu, assert_close
from test_gpu_real_integer import general

pytestmark = pytest.mark.gpu

INTEGRALS = {"bubble_m0": (lambda: w.bubble(0, "s"), -1, [[9.0]]),
             "bubble_m1": (lambda: w.bubble(1, "s"), 0, [[9.0]]),
             "triangle_m0": (lambda: w.triangle_one_offshell(0, "s"), -2, [[7.0]]),
             "triangle_m1": (lambda: w.triangle_one_offshell(1, "s"), 0, [[7.0]]),
             "box_m0": (lambda: w.box_massless(deform=True), -2, [[12.0, -3.0], [6.5, -2.25]]),
             "box_m1": (w.box_massive, 0, [[12.0, -3.0]])}


def _oracle(I, sp, inv, m, lo, nord, transform):
    sec = I.sectors[sp["sector"]]
    _, z = lattice_for(sp["n"], sec.d)
    delta = np.zeros((m, sec.d)) if sp["flags"] else oracle.shifts(11, sp["stream"], m, sec.d)
    view = oracle.SectorView(I, sp["sector"], inv, sp["lambda"], transform=transform)
    o, a, _, c = oracle.shift_sums(view, sp["n"], z, delta, lo, nord, with_cond=True)
    return o, a, c


@pytest.mark.parametrize("name", sorted(INTEGRALS))
@pytest.mark.parametrize("transform,mixed,n,block,flags", [
    (0, False, 1009, 0, 0), (0, False, 10007, 128, 0), (0, True, 2003, 256, 0), (1, False, 4001, 256, 0),
    (2, True, 1259, 128, 0), (0, False, 1009, 0, qmc.QMC_JOB_UNSHIFTED)])
def test_same_sums_as_the_general_kernel(name, transform, mixed, n, block, flags):
    """Both evaluate one formula in FP64 (the same FP32 products in mixed
    precision): the bar is twice the parity bar, 2e-12 max(|Q|, A) + 6e-16 C,
    with A and C from the oracle."""
    build, lo, kin = INTEGRALS[name]
    I = build()
    g = Gpu(transform=transform, block=block,
            precision=qmc.QMC_PRECISION_MIXED if mixed else qmc.QMC_PRECISION_FP64)
    try:
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array(kin))
        m = 1 if flags else 2
        specs = [dict(integral_id=iid, sector=s, point=p, shifts=m, n=n, seed=11, stream=p * 20 + s, flags=flags,
                      **{"lambda": 0.6}) for p in range(len(kin)) for s in range(len(I.sectors))]
        gid = g.load(general(I, Fraction(1, 10 ** 250)))
        for hi in (0, 1):
            nord = hi - lo + 1
            a, fa, _ = g.eval(iid, specs, lo, nord)
            if mixed:
                b, fb, _ = g.eval(iid, specs, lo, 2 - lo if hi == 0 else 1 - lo)
                nb = 2 - lo if hi == 0 else 1 - lo
            else:
                b, fb, _ = g.eval(gid, [dict(sp, integral_id=gid) for sp in specs], lo, nord)
                nb = nord
            assert fa == fb
            a = a.reshape(len(specs), m, nord, 2)
            b = b.reshape(len(specs), m, nb, 2)
            for i, sp in enumerate(specs):
                o, A, C = _oracle(I, sp, kin[sp["point"]], m, lo, nord, transform)
                bar = 2e-12 * np.maximum(np.abs(o), A[..., None]) + 6e-16 * C[..., None]
                k = min(nb, nord)
                err, bar = np.abs(a[i][:, :k] - b[i][:, :k]), bar[:, :k]
                assert np.all(err <= bar), (sp, hi, float(np.max(err / bar)))
    finally:
        g.close()


def test_higher_degree_stays_on_the_general_kernel():
    """A sector whose F has total degree 3 beside one of degree 2: one plan,
    two launches, both match the oracle."""
    head = "qmc-sectors 1\nname toy\nloops 1 propagators 4 dim 4\ninvariants 2 s t\nprefactor 0 1 1.0 0.0\nnsectors 2\n"
    body = ("a 0 0\nb 0.0 0.0\nU 0.0 2.0 2\n0 0 1.0 0.0 0.0\n1 0 1.0 0.0 0.0\n"
            "F -2.0 -1.0 3\n0 0 1.0 0.0 0.0\n1 1 0.0 -1.0 0.0\n{e} 1.0 0.0 0.0\n")
    text = head + "sector 0 d 2 deform 1\n" + body.format(e="2 0") + "sector 1 d 2 deform 1\n" + body.format(e="2 1") + "end\n"
    I = Integral.from_text(text)
    g = Gpu()
    try:
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array([[3.0, -1.0]]))
        specs = [dict(integral_id=iid, sector=s, point=0, shifts=2, n=2003, seed=11, stream=s, flags=0,
                      **{"lambda": 0.3}) for s in (0, 1)]
        out, _, _ = g.eval(iid, specs, 0, 1)
        for i, sp in enumerate(specs):
            o, A, C = _oracle(I, sp, [3.0, -1.0], 2, 0, 1, 0)
            assert_close(out.reshape(2, 2, 1, 2)[i], o, A, C, what=f"sector {i}")
    finally:
        g.close()
