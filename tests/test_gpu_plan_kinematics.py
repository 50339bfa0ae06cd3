"""A plan run after its kinematics were replaced (GPU): by other values it
follows them, on the d <= 6 evaluators too; by fewer points, or by points with
another number of invariants, the run is refused, and runs again when they fit."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads as w

from parity import Gpu, assert_close, oracle_sums
from test_gpu_real_integer import general

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("build,kin", [(w.box_massless, [-3.0, -2.0]), (lambda: w.box_massive(), [12.0, -3.0])])
def test_kinematics_that_do_not_fit_the_plan_are_refused(build, kin, graph):
    I, lo, nord = build(), -2, 3
    g = Gpu()
    try:
        iid = g.load(I)
        two, one = np.array([kin, [1.1 * x for x in kin]]), np.array([kin])
        qmc.qmc_set_kinematics(g.ctx, two)
        jobs, nj = qmc.make_jobs(qmc.jobs_for_integral(iid, len(I.sectors), 2, 1009, 2, seed=5, lam=0.5))
        plan = qmc.qmc_plan_create(g.ctx, jobs, nj, lo, nord)
        qmc.qmc_plan_use_graph(g.ctx, plan, graph)
        qmc.qmc_plan_run(g.ctx, plan)
        ref = qmc.qmc_plan_results(g.ctx, plan)[0].copy()
        for bad in (one, np.zeros((2, 1)), np.zeros((0, 2))):
            qmc.qmc_set_kinematics(g.ctx, bad)
            for _ in range(2):
                with pytest.raises(qmc.QmcError) as e:
                    qmc.qmc_plan_run(g.ctx, plan)
                assert e.value.code == -1
        for good in (two, np.concatenate([two, one])):
            qmc.qmc_set_kinematics(g.ctx, good)
            qmc.qmc_plan_run(g.ctx, plan)
            assert np.array_equal(qmc.qmc_plan_results(g.ctx, plan)[0], ref)
        qmc.qmc_plan_destroy(plan)
    finally:
        g.close()


def test_plans_without_invariants_run_on_any_kinematics():
    I = w.triangle_massive()
    g = Gpu()
    try:
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array([[-3.0, -2.0]]))
        jobs, nj = qmc.make_jobs(qmc.jobs_for_integral(iid, len(I.sectors), 1, 1009, 2, seed=5))
        plan = qmc.qmc_plan_create(g.ctx, jobs, nj, 0, 1)
        seen = []
        for kin in (np.array([[-3.0, -2.0]]), np.zeros((1, 0)), np.zeros((0, 0))):
            qmc.qmc_set_kinematics(g.ctx, kin)
            qmc.qmc_plan_run(g.ctx, plan)
            seen.append(qmc.qmc_plan_results(g.ctx, plan)[0].copy())
        assert np.array_equal(seen[0], seen[1]) and np.array_equal(seen[0], seen[2])
        qmc.qmc_plan_destroy(plan)
    finally:
        g.close()


@pytest.mark.parametrize("graph", [False, True])
def test_changed_kinematics_of_a_two_loop_plan(graph):
    """d <= 6: tiles of 384 threads cut again for the general kernel's 128 where
    the new kinematics leave the integer evaluator's range, and back."""
    I = w.double_box_massless()
    g = Gpu()
    try:
        iid = g.load(I)
        near, far = np.array([[-3.0, -1.0]]), np.array([[-3000.0, -1.0]])
        qmc.qmc_set_kinematics(g.ctx, near)
        specs = [dict(integral_id=iid, sector=s, point=0, shifts=2, n=1009, seed=11, stream=s)
                 for s in range(0, len(I.sectors), 25)]
        jobs, nj = qmc.make_jobs(specs)
        plan = qmc.qmc_plan_create(g.ctx, jobs, nj, -4, 5)
        qmc.qmc_plan_use_graph(g.ctx, plan, graph)
        seen = []
        for kin in (near, far, near):
            qmc.qmc_set_kinematics(g.ctx, kin)
            qmc.qmc_plan_run(g.ctx, plan)
            seen.append(qmc.qmc_plan_results(g.ctx, plan)[0].copy())
            for sp, x in zip(specs, seen[-1].reshape(len(specs), 2, 5, 2)):
                o, a, c = oracle_sums(I, sp["sector"], kin[0], 1009, 2, 11, sp["stream"], -4, 5)
                assert_close(x, o, a, c, what=f"{kin} sector {sp['sector']}")
        assert np.array_equal(seen[0], seen[2])
        qmc.qmc_plan_destroy(plan)
    finally:
        g.close()


@pytest.mark.parametrize("graph", [False, True])
def test_a_plan_after_another_integral_was_loaded(graph):
    g = Gpu()
    try:
        I = w.box_massless()
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array([[-3.0, -2.0]]))
        jobs, nj = qmc.make_jobs(qmc.jobs_for_integral(iid, len(I.sectors), 1, 1009, 2, seed=5))
        plan = qmc.qmc_plan_create(g.ctx, jobs, nj, -2, 3)
        qmc.qmc_plan_use_graph(g.ctx, plan, graph)
        qmc.qmc_plan_run(g.ctx, plan)
        ref = qmc.qmc_plan_results(g.ctx, plan)[0].copy()
        for build in (w.double_box_massless, w.box_massive):
            g.load(build())
            qmc.qmc_plan_run(g.ctx, plan)
            assert np.array_equal(qmc.qmc_plan_results(g.ctx, plan)[0], ref)
        qmc.qmc_plan_destroy(plan)
    finally:
        g.close()


@pytest.mark.parametrize("opts", [{}, {"ppt": 5}, {"block": 256}])
@pytest.mark.parametrize("build,lo,n,step", [(w.box_massless, -2, 1009, 1), (w.box_massless, -2, 20011, 1),
                                             (w.double_box_massless, -4, 1009, 25)])
def test_general_kernel_with_its_own_tiles(build, lo, n, step, opts):
    """Where new kinematics take a plan to the general kernel it has the tiles that
    a plan of the general kernel has: the same bits as one (whose F carries a
    negligible negative monomial), also when it comes back a second time."""
    I = build()
    g = Gpu(**opts)
    try:
        iid, gid = g.load(I), g.load(general(I, Fraction(-1, 10 ** 250)))
        near, far = np.array([[-3.0, -1.0]]), np.array([[-3000.0, -1.0]])
        specs = [dict(integral_id=iid, sector=s, point=0, shifts=2, n=n, seed=11, stream=s)
                 for s in range(0, len(I.sectors), step)]
        jobs, nj = qmc.make_jobs(specs)
        qmc.qmc_set_kinematics(g.ctx, near)
        plan = qmc.qmc_plan_create(g.ctx, jobs, nj, lo, 1 - lo)
        qmc.qmc_set_kinematics(g.ctx, far)
        ref, _, rc = g.eval(gid, [dict(sp, integral_id=gid) for sp in specs], lo, 1 - lo)
        assert rc == 0
        for kin in (far, near, far):
            qmc.qmc_set_kinematics(g.ctx, kin)
            qmc.qmc_plan_run(g.ctx, plan)
            got = qmc.qmc_plan_results(g.ctx, plan)[0]
            assert np.array_equal(got, ref) == (kin is far)
        qmc.qmc_plan_destroy(plan)
    finally:
        g.close()
