"""Paths of the evaluators on integers that the built-in integrals do not reach
(GPU): mixed-precision deformed sectors with F of degree 3 to 6 and couplings
(second derivatives from the monomial tables), against the general mixed kernel
(which serves a window up to eps^2) and the oracle; and tiles of any number of
points per thread, against the general kernels."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads as w
from paper_2305_19768_gb300.inputs.integral import Integral

from parity import Gpu
from test_gpu_deformed_quadratic import _oracle
from test_gpu_mixed import MIX_CTOL, MIX_RTOL
from test_gpu_real_integer import _compare, _specs, general

pytestmark = pytest.mark.gpu

# d, a, b, U, F (coefficient, coefficient of s): F of degree 3 to 4 in a variable
# or two, every pair of variables coupled by non-constant second derivatives
SECTORS = {
    "d1": (1, [-1], [-2], {(0,): (1, 0), (1,): (1, 0)}, {(0,): (1, 0), (1,): (0, -1), (3,): (1, 0)}),
    "d2": (2, [0, 1], [1, -1], {(0, 0): (1, 0), (1, 1): (2, 0)},
           {(0, 0): (1, 0), (1, 1): (0, -1), (2, 1): (1, 0), (0, 3): (0.5, 0)}),
    "d3": (3, [0, 0, 0], [0, 0, 0], {(0, 0, 0): (1, 0), (1, 0, 1): (1, 0)},
           {(0, 0, 0): (2, 0), (1, 1, 1): (0, -1), (2, 0, 1): (1, 0), (0, 2, 2): (0.5, 0), (1, 0, 0): (1, 0)}),
    "d3_pole": (3, [0, -1, 2], [0, -2, 1], {(0, 0, 0): (1, 0), (0, 1, 1): (1, 0)},
                {(0, 0, 0): (1, 0), (1, 1, 0): (1, 0), (0, 1, 2): (0, -1), (3, 0, 1): (0.5, 0), (0, 0, 1): (1, 0)}),
}


def _integral(name):
    d, a, b, U, F = SECTORS[name]
    out = ["qmc-sectors 1", "name toy", f"loops 1 propagators {d + 1} dim 4", "invariants 1 s",
           "prefactor 0 1 1.0 0.0", "nsectors 1", f"sector 0 d {d} deform 1", "a " + " ".join(map(str, a)),
           "b " + " ".join(f"{x}.0" for x in b)]
    for tag, P, e0, e1 in (("U", U, 1.0, 2.0), ("F", F, -2.0, -1.0)):
        out.append(f"{tag} {e0} {e1} {len(P)}")
        out += [" ".join(map(str, e)) + f" {c[0]} {c[1]}" for e, c in P.items()]
    return Integral.from_text("\n".join(out + ["end"]) + "\n")


@pytest.mark.parametrize("name", sorted(SECTORS))
@pytest.mark.parametrize("transform,n,s", [(0, 1009, 3.0), (1, 4001, 0.75), (2, 2003, -2.0)])
def test_mixed_deformed_sectors_of_higher_degree(name, transform, n, s):
    """Against the general kernel at the bar of test_gpu_deformed_quadratic (the
    FP32 products are the same), against the oracle at the mixed one."""
    I, m, lo = _integral(name), 2, -1
    g = Gpu(transform=transform, precision=qmc.QMC_PRECISION_MIXED)
    try:
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array([[s]]))
        sp = dict(integral_id=iid, sector=0, point=0, shifts=m, n=n, seed=11, stream=1, flags=0, **{"lambda": 0.2})
        b, fb, _ = g.eval(iid, [sp], lo, 4)
        o, A, C = _oracle(I, sp, [s], m, lo, 3, transform)
        for nord in (2, 3):
            a, fa, _ = g.eval(iid, [sp], lo, nord)
            a, ref = a.reshape(m, nord, 2), b.reshape(m, 4, 2)[:, :nord]
            assert fa == fb
            scale, mass = np.maximum(np.abs(o), A[..., None])[:, :nord], C[..., None][:, :nord]
            assert np.all(np.abs(a - ref) <= 2e-12 * scale + 6e-16 * mass)
            assert np.all(np.abs(a - o[:, :nord]) <= MIX_RTOL * scale + MIX_CTOL * mass)
    finally:
        g.close()


@pytest.mark.parametrize("ppt", [1, 5, 32])
@pytest.mark.parametrize("n", [1009, 16001])
@pytest.mark.parametrize("name,mixed", [("box", False), ("box", True), ("double_box", False), ("box_massive", False)])
def test_points_per_thread(name, mixed, n, ppt):
    """Tiles that end inside, at and beyond the lattice (256 or 384 threads of ppt
    points) give the general kernels' sums."""
    build, lo, kin = {"box": (w.box_massless, -2, [-3.0, -2.0]), "double_box": (w.double_box_massless, -4, [-3.0, -1.0]),
                      "box_massive": (w.box_massive, 0, [12.0, -3.0])}[name]
    I, m, nord = build(), 2, 1 - lo
    g = Gpu(ppt=ppt, precision=qmc.QMC_PRECISION_MIXED if mixed else qmc.QMC_PRECISION_FP64)
    try:
        iid = g.load(I)
        gid = g.load(general(I, Fraction(1 if name == "box_massive" else -1, 10 ** 250)))
        qmc.qmc_set_kinematics(g.ctx, np.array([kin]))
        specs = [dict(sp, **{"lambda": 0.6}) for sp in _specs(iid, I, name, 1, n, m)]
        if name == "double_box":
            specs = specs[::4]
        a, fa, ra = g.eval(iid, specs, lo, nord)
        b, fb, rb = g.eval(gid, [dict(sp, integral_id=gid) for sp in specs], lo, nord)
        assert ra == rb == 0 and fa == fb
        if name != "box_massive":
            _compare(I, specs, a, b, [kin], m, lo, nord, 0)
        else:
            a, b = a.reshape(len(specs), m, nord, 2), b.reshape(len(specs), m, nord, 2)
            for x, y, sp in zip(a, b, specs):
                o, A, C = _oracle(I, sp, kin, m, lo, nord, 0)
                assert np.all(np.abs(x - y) <= 2e-12 * np.maximum(np.abs(o), A[..., None]) + 6e-16 * C[..., None])
    finally:
        g.close()
