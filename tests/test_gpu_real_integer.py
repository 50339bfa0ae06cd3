"""The integer evaluator of the real classes (csrc/qmc_real.cuh, GPU): against
the general kernels on everything it accepts (they run where a coefficient is
negative), at the edge of its coefficient rule against the
oracle, and its fall-back when a plan's kinematics change."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads as w
from paper_2305_19768_gb300.inputs.lattice import lattice_for

from parity import Gpu, assert_close, oracle_sums

pytestmark = pytest.mark.gpu

INTEGRALS = {"triangle": (w.triangle_massive, 0, [[]]),
             "box": (w.box_massless, -2, [[-3.0, -2.0], [-2.5, -1.25]]),
             "bubble_t": (lambda: w.bubble(0, "t", deform=False), 0, [[-2.0]]),
             "double_box": (w.double_box_massless, -4, [[-3.0, -1.0]]),
             "double_box_geometric": (lambda: w.double_box_massless(method="geometric"), -4, [[-3.0, -1.0]])}


def _specs(iid, I, name, npts, n, m, flags=0):
    step = 1 if len(I.sectors) < 20 else 9
    return [dict(integral_id=iid, sector=s, point=p, shifts=m, n=n, seed=11, stream=p * len(I.sectors) + s,
                 flags=flags) for p in range(npts) for s in range(0, len(I.sectors), step)]


def general(I, c):
    """The integral with one more monomial c t_1^4 .. t_d^4 in each sector's F,
    far below rounding: a negative one keeps a real sector off the integer
    evaluator, and its degree a deformed one off the quadratic evaluator."""
    J = type(I).from_text(I.to_text())
    for s in J.sectors:
        s.F._acc((4,) * s.d, (c,) + (0,) * len(I.invariants))
    return J


def _corner_mass(I, sp, inv, m, lo, nord, transform):
    """C of the job's sums (parity.py), from the oracle: [m][nord]"""
    sec = I.sectors[sp["sector"]]
    _, z = lattice_for(sp["n"], sec.d)
    delta = np.zeros((m, sec.d)) if sp["flags"] else oracle.shifts(11, sp["stream"], m, sec.d)
    view = oracle.SectorView(I, sp["sector"], inv, transform=transform)
    return oracle.shift_sums(view, sp["n"], z, delta, lo, nord, with_cond=True)[3]


@pytest.mark.parametrize("name", sorted(INTEGRALS))
@pytest.mark.parametrize("transform,mixed,n,block,flags", [
    (0, False, 1009, 0, 0), (0, False, 16001, 256, 0), (0, True, 2003, 0, 0), (1, False, 4001, 0, 0),
    (2, False, 1259, 128, 0), (0, False, 1009, 0, qmc.QMC_JOB_UNSHIFTED)])
def test_same_sums_as_the_general_kernels(name, transform, mixed, n, block, flags):
    """FP64 evaluations of one formula differ by some u of the cancelling corner
    terms' mass C (parity.py): the bar is 1e-12 |Q| + 6e-16 C, both sides'
    allowance, with C from the oracle; FP32 products are the
    same on both sides, so the mixed bar is the same."""
    build, lo, kin = INTEGRALS[name]
    I = build()
    g = Gpu(transform=transform, block=block,
            precision=qmc.QMC_PRECISION_MIXED if mixed else qmc.QMC_PRECISION_FP64)
    try:
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array(kin))
        m = 1 if flags else 3
        specs = _specs(iid, I, name, len(kin), n, m, flags)
        gid = g.load(general(I, Fraction(-1, 10 ** 250)))
        for hi in (0, 1) if I.sectors[0].d <= 3 else (0,):
            nord = hi - lo + 1
            a, _, ra = g.eval(iid, specs, lo, nord)
            b, _, rb = g.eval(iid, [dict(sp, integral_id=gid) for sp in specs], lo, nord)
            assert ra == 0 and rb == 0
            _compare(I, specs, a, b, kin, m, lo, nord, transform)
    finally:
        g.close()


def _compare(I, specs, a, b, kin, m, lo, nord, transform):
    a, b = a.reshape(len(specs), m, nord, 2), b.reshape(len(specs), m, nord, 2)
    for sp, x, y in zip(specs, a, b):
        C = _corner_mass(I, sp, kin[sp["point"]], m, lo, nord, transform)
        assert np.all(np.abs(x - y) <= 1e-12 * np.abs(y).max(axis=(0, 2), keepdims=True) + 6e-16 * C[..., None])


@pytest.mark.parametrize("ratio", [10.0, 100.0, 1000.0])
def test_coefficient_rule_edges_match_the_oracle(ratio):
    """Up to a sum of coefficients of 128 c0 the fixed-point polynomials hold
    FP64's precision; beyond it the general kernel runs: both within the bar."""
    I = w.box_massless()
    g = Gpu()
    try:
        iid = g.load(I)
        for kin in ([-ratio, -1.0], [-1.0, -ratio], [-1e-3, -1e-3 * ratio]):
            qmc.qmc_set_kinematics(g.ctx, np.array([kin]))
            specs = _specs(iid, I, "box", 1, 1009, 2)
            out, _, rc = g.eval(iid, specs, -2, 3)
            assert rc == 0
            for i, sp in enumerate(specs):
                o, a, c = oracle_sums(I, sp["sector"], kin, 1009, 2, 11, sp["stream"], -2, 3)
                assert_close(out.reshape(len(specs), 2, 3, 2)[i], o, a, c, what=f"{kin} sector {sp['sector']}")
    finally:
        g.close()


@pytest.mark.parametrize("graph", [False, True])
def test_changed_kinematics_of_a_plan(graph):
    """A plan made where its jobs qualify runs the general kernel once they do
    not (and the integer one again when they do)."""
    I = w.box_massless()
    g = Gpu()
    try:
        iid = g.load(I)
        near, far = np.array([[-3.0, -2.0]]), np.array([[-3000.0, -1.0]])
        qmc.qmc_set_kinematics(g.ctx, near)
        specs = _specs(iid, I, "box", 1, 2003, 2)
        jobs, nj = qmc.make_jobs(specs)
        plan = qmc.qmc_plan_create(g.ctx, jobs, nj, -2, 3)
        qmc.qmc_plan_use_graph(g.ctx, plan, graph)
        seen = []
        for kin in (near, far, near):
            qmc.qmc_set_kinematics(g.ctx, kin)
            qmc.qmc_plan_run(g.ctx, plan)
            seen.append(qmc.qmc_plan_results(g.ctx, plan)[0].copy())
            for sp, x in zip(specs, seen[-1].reshape(len(specs), 2, 3, 2)):
                o, a, c = oracle_sums(I, sp["sector"], kin[0], 2003, 2, 11, sp["stream"], -2, 3)
                assert_close(x, o, a, c, what=f"{kin} sector {sp['sector']}")
        assert np.array_equal(seen[0], seen[2])
        qmc.qmc_plan_destroy(plan)
    finally:
        g.close()
