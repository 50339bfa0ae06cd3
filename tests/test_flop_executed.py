"""The executed FP64 counts of the evaluators on integers (flops.py) against
counts made by hand, and the rules by which they are chosen. The same walk of
the massive box's operations gives 68 instructions, what the profiler counts
(profiles/qmc_deformed_kernel_box1L_massive_batch.md)."""
import pytest

from paper_2305_19768_gb300 import flops as F
from paper_2305_19768_gb300.inputs import workloads as w


def test_massive_box_by_hand():
    # gradient: 3 squares twice, 3 pairs twice, FMAs: 24; y: 3; M: 6
    # minors 3 x 3; det M0 c12: 1, two couplings 3 each, the third 1 + 2 (the doubling is free)
    # Jacobian: p0 p1: 1; re: 2 + 3 + 3; im: three FMAs, two products
    # F: re 3 FMAs: 6; A_jj y_j / 2 + couplings: (1 + 4) + (1 + 2) + 1; -y q: 6; im: 1 + 2 + 2
    # F^-2: |F|^2 3, conj(F)^2 4, product 6; accumulation 4
    hand = 24 + 3 + 6 + 9 + 10 + 1 + 8 + 8 + 6 + 9 + 6 + 5 + 13 + 4
    assert hand == 112
    assert F.executed_workload(w.box_massive(), [10.0, -3.0], 0, 1).fp64 == hand


def test_one_pole_by_hand():
    # d <= 3, one singular variable, sums up to eps^0: b / t and b ln t 2; corner
    # series B and B L: 1; fold: one difference, one FMA: 3; two accumulations 4
    I = w.box_massless()
    s = next(s for s in I.sectors if sum(1 for a in s.a if a <= -1) == 1)
    reg = sum(1 for a, b in zip(s.a, s.b) if a > 0 or (a > -1 and b))
    logs = any(a > -1 and b for a, b in zip(s.a, s.b))
    assert F.executed_work(s, [-3.0, -2.0], -2, 3).fp64 == 2 + 2 * reg + (1 if logs else 0) + 1 + 3 + 4


@pytest.mark.parametrize("build,lo,nord,inv", [(w.box_massless, -2, 3, [-3.0, -2.0]),
                                               (w.double_box_massless, -4, 5, [-3.0, -1.0]),
                                               (w.box_massive, 0, 1, [10.0, -3.0]),
                                               (lambda: w.box_massless(deform=True), -2, 3, [7.0, -2.5])])
def test_fewer_than_the_general_formulation(build, lo, nord, inv):
    I = build()
    assert all(F.takes_integer_evaluator(s, inv, lo + nord - 1) for s in I.sectors)
    assert 0 < F.executed_workload(I, inv, lo, nord).fp64 < F.workload_work(I, lo, nord).fp64


def test_the_rules():
    box, two = w.box_massless(), w.double_box_massless()
    far = [-3000.0, -1.0]
    assert not all(F.takes_integer_evaluator(s, far, 0) for s in box.sectors)
    assert not F.takes_integer_evaluator(box.sectors[0], [3.0, -2.0], 0)      # a negative coefficient
    assert F.takes_integer_evaluator(box.sectors[0], [-3.0, -2.0], 1)
    assert not F.takes_integer_evaluator(box.sectors[0], [-3.0, -2.0], 2)
    assert not F.takes_integer_evaluator(two.sectors[0], [-3.0, -1.0], 1)
    s = next(s for s in box.sectors if not F.takes_integer_evaluator(s, far, 0))
    assert F.executed_work(s, far, -2, 3).fp64 == F.sector_work(s, -2, 3).fp64
    d2 = w.box_massless_d2()
    assert F.executed_workload(d2, [-3.0, -2.0], -2, 3) is None
    assert F.executed_workload(w.box_massive(), [10.0, -3.0], 0, 1, mixed=True) is None
