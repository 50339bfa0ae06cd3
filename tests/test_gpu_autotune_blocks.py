"""The autotuner on classes whose jobs run the evaluators with one block size
(GPU): that size is reported, and a class with general jobs gets a size that its
kernels have."""
import numpy as np
import pytest

from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads as w

from parity import Gpu

pytestmark = pytest.mark.gpu

PPT = (1, 2, 4, 8, 16, 32)


@pytest.mark.parametrize("build,lo,kin,expect", [
    (w.box_massless, -2, [-3.0, -2.0], {256}),                     # real d <= 3, integers
    (w.box_massive, 0, [12.0, -3.0], {256}),                       # deformed d <= 3
    (w.double_box_massless, -4, [-3.0, -1.0], {384}),              # real d <= 6, integers
    (w.box_massless, -2, [-3000.0, -1.0], {128, 256}),             # general: coefficients too far apart
    (w.double_box_massless, -4, [-3000.0, -1.0], {128})])
def test_reported_block(build, lo, kin, expect):
    I = build()
    g = Gpu()
    try:
        iid = g.load(I)
        qmc.qmc_set_kinematics(g.ctx, np.array([kin]))
        jobs, nj = qmc.make_jobs(qmc.jobs_for_integral(iid, len(I.sectors), 1, 1009, 2, seed=5, lam=0.5))
        ref = qmc.qmc_eval_jobs(g.ctx, jobs, nj, lo, 1 - lo, nj * 2 * (1 - lo) * 2)
        block, ppt = qmc.qmc_autotune(g.ctx, jobs, nj, lo, 1 - lo)
        seen = {b for b in block if b}
        assert seen and seen <= expect
        assert all(p in PPT for b, p in zip(block, ppt) if b)
        got = qmc.qmc_eval_jobs(g.ctx, jobs, nj, lo, 1 - lo, nj * 2 * (1 - lo) * 2)
        assert np.max(np.abs(got - ref)) <= 1e-12 * np.abs(ref).max()
    finally:
        g.close()
