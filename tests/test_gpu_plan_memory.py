"""A plan's one device allocation (GPU): results on both sides of the size up
to which they come back in one copy with the status, several class launches in
one plan, and what a plan says before its first run."""
import numpy as np
import pytest

from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads as w
from parity import Gpu

pytestmark = pytest.mark.gpu


def _run(g, specs, lo, nord, out=None):
    jobs, total = qmc.make_jobs(specs)
    p = qmc.qmc_plan_create(g.ctx, jobs, len(specs), lo, nord)
    try:
        before, fails, rc = qmc.qmc_plan_results(g.ctx, p)
        assert rc == 0 and fails == 0
        assert not qmc.qmc_plan_job_failures(g.ctx, p, len(specs)).any()
        res = []
        for _ in range(2):   # the second run finds queues and counts as the first did
            qmc.qmc_plan_run(g.ctx, p)
            o, fails, rc = qmc.qmc_plan_results(g.ctx, p)
            assert rc == 0 and fails == 0
            res.append(o)
        assert np.array_equal(res[0], res[1])
        return res[0]
    finally:
        qmc.qmc_plan_destroy(p)


@pytest.mark.parametrize("shifts", [1, 2047, 2048, 2049])
def test_results_in_one_copy_or_two(shifts):
    """2048 complex sums come with the status, 2049 apart; shift i's sum is the
    same bits whatever the number of shifts."""
    g = Gpu(ppt=4)   # one summation order whatever the plan
    try:
        I = w.triangle_massive()
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.zeros((1, 0)))
        one = [dict(integral_id=iid, sector=0, point=0, n=1009, seed=5, stream=3)]
        o = _run(g, [dict(one[0], shifts=shifts)], 0, 1)
        ref = _run(g, [dict(one[0], shifts=2500)], 0, 1)
        assert o.shape[0] == shifts * (ref.shape[0] // 2500)
        assert np.array_equal(o, ref[:o.shape[0]])
    finally:
        g.close()


def test_several_classes_in_one_plan():
    """Jobs of two classes in one plan give the bits of two plans."""
    g = Gpu(ppt=4)   # one summation order whatever the plan
    try:
        a = g.load(w.box_massless())
        b = g.load(w.box_massive(1))
        qmc.qmc_set_kinematics(g.ctx, np.array([[-3.0, -2.0]]))
        sa = [dict(integral_id=a, sector=s, point=0, shifts=3, n=1009, seed=5, stream=s) for s in range(2)]
        sb = [dict(integral_id=b, sector=s, point=0, shifts=5, n=1009, seed=5, stream=s,
                   **{"lambda": 0.25}) for s in range(3)]
        both = _run(g, [sb[0], sa[0], sb[1], sa[1], sb[2]], -2, 3)
        ra, rb = _run(g, sa, -2, 3), _run(g, sb, -2, 3)
        na, nb = ra.shape[0] // 2, rb.shape[0] // 3
        cut = np.cumsum([0, nb, na, nb, na, nb])
        parts = [both[cut[i]:cut[i + 1]] for i in range(5)]
        assert np.array_equal(np.concatenate(parts[1::2]), ra)
        assert np.array_equal(np.concatenate(parts[0::2]), rb)
    finally:
        g.close()
