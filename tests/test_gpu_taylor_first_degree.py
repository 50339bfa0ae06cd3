"""The first-degree Taylor subtraction written out (eval_real_taylor1, sums up
to eps^0, GPU) against the loops for any degree, which serve a window up to
eps^1: the orders that both give have the same bits, since the written-out form
takes the loops' roundings step by step."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads as w

from parity import Gpu
from test_oracle_pins import _toy_integral

pytestmark = pytest.mark.gpu

# one variable; two with p = (2, 1), (1, 2), (2, 2); the singular variables not the
# first ones; powers 1 to 4, also of the singular variables; exponents of the
# base that are integers, fractions, zero; regular factors t^a, t^(b eps)
SECTORS = {
    "p2": (1, [-2], ["5/4"], {(0,): 1, (1,): 2, (2,): 3, (4,): "1/2"}, "1/2", 2, {(0,): 2, (1,): 1}, -2, -1),
    "p2_third": (3, [2, 0, -2], ["1/2", "0", "-2"], {(0, 0, 0): 1, (3, 0, 1): 2, (0, 4, 0): 1, (1, 2, 1): 3}, 2, 0,
                 {(0, 0, 0): 1, (0, 0, 3): 1, (2, 1, 0): 5}, "-3/2", -1),
    "p21": (2, [-2, -1], ["5/4", "-1/2"], {(0, 0): 1, (1, 0): 1, (1, 1): 2, (0, 2): 1}, 0, 2,
            {(0, 0): 2, (1, 0): 1, (0, 1): 1}, -3, -1),
    "p12": (3, [-1, 1, -2], ["1", "1/2", "-2"], {(0, 0, 0): 1, (1, 0, 0): 1, (0, 1, 0): 2, (1, 1, 1): "1/2"}, -1, 2,
            {(0, 0, 0): 2, (1, 0, 1): 1, (0, 2, 0): "1/2", (0, 3, 1): 1}, -2, -1),
    "p22": (3, [0, -2, -2], ["0", "3/4", "-1/2"], {(0, 0, 0): 1, (0, 1, 1): 1, (1, 1, 0): 2, (2, 0, 1): 1, (0, 2, 0): 1},
            2, 3, {(0, 0, 0): 3, (0, 1, 0): 1, (0, 0, 1): 2, (1, 1, 1): 1}, -3, 0),
}


def _integral(name):
    if name == "box_d2":
        return w.box_massless_d2(), [[-3.0, -2.0]]
    d, a, b, U, u0, u1, F, f0, f1 = SECTORS[name]
    fr = lambda v: {e: Fraction(str(c)) for e, c in v.items()}
    return _toy_integral(d, a, [Fraction(x) for x in b], fr(U), u0=Fraction(str(u0)), u1=Fraction(str(u1)),
                         Fterms=fr(F), f0=Fraction(str(f0)), f1=Fraction(str(f1))), None


@pytest.mark.parametrize("transform,block", [(0, 0), (1, 256)])
@pytest.mark.parametrize("n,shifts", [(1009, 3), (16001, 2)])
@pytest.mark.parametrize("name", sorted(SECTORS) + ["box_d2"])
def test_same_bits_as_the_loops(name, n, shifts, transform, block):
    g = Gpu(transform=transform, block=block)
    try:
        I, kin = _integral(name)
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array(kin) if kin else np.zeros((0, 0)))
        specs = [dict(integral_id=iid, sector=s, point=0, shifts=shifts, n=n, seed=3, stream=s)
                 for s in range(len(I.sectors))]
        lo = -2
        a, _, ra = g.eval(iid, specs, lo, 1 - lo)
        b, _, rb = g.eval(iid, specs, lo, 2 - lo)
        assert ra == 0 and rb == 0
        a = a.reshape(len(specs), shifts, 1 - lo, 2)
        b = b.reshape(len(specs), shifts, 2 - lo, 2)
        assert np.array_equal(a, b[:, :, :1 - lo])
        assert np.abs(a[..., 0]).max() > 0
    finally:
        g.close()
