"""qmc_integrate over ranks whose lattices end below the default cap (GPU): the
tiles, and with them the order of summation, follow from the whole pass, so
that two ranks give one rank's result bit for bit. The ranks are processes
whose kernels never wait on each other (the exchange runs on the host)."""
import os
import socket

import numpy as np
import pytest

from paper_2305_19768_gb300 import dist as qdist
from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads as w

pytestmark = pytest.mark.gpu

KIN = {"box": [[-3.0, -2.0], [-5.0, -1.0], [-2.0, -7.0]], "box_massive": [[10.0, -3.0], [7.0, -2.0], [15.0, -5.0]]}


def _worker(rank, port, world, name, most, median, result_dir):
    import torch.distributed as dist

    dist.init_process_group("gloo", init_method=f"tcp://127.0.0.1:{port}", rank=rank, world_size=world)
    ctx = qmc.qmc_create(0, keep_shift_sums=1, shifts=8, max_points=most, lambda_=0.5 if name == "box_massive" else 0.0,
                         **({"lattice_candidates": 5} if median else {}))
    try:
        qmc.load_lattice_table(ctx)
        I, lo, nord = (w.box_massless(), -2, 3) if name == "box" else (w.box_massive(), 0, 1)
        iid = qmc.qmc_load_sectors_mem(ctx, I.to_text())
        qmc.qmc_set_kinematics(ctx, np.array(KIN[name]))
        if world > 1:
            qdist.set_ranks(ctx)
        val, err, info, rc = qmc.qmc_integrate(ctx, [iid], epsrel=1e-14, lowest_order=lo, norders=nord, npoints=3,
                                               check=False)
        sums, _, n = qmc.qmc_per_shift_sums(ctx, iid)
        if rank == 0:
            np.savez(os.path.join(result_dir, f"g{world}.npz"), val=val, err=err, sums=sums, n=n, rc=rc,
                     evals=info["evaluations"], iters=info["iterations"])
    finally:
        qmc.qmc_destroy(ctx)
        dist.destroy_process_group()


@pytest.mark.parametrize("name,most,median", [("box", 100003, False), ("box", 40009, True), ("box_massive", 10007, False)])
def test_two_ranks_equal_one_on_small_lattices(tmp_path, name, most, median):
    import torch.multiprocessing as mp

    res = {}
    for world in (1, 2):
        with socket.socket() as s:
            s.bind(("127.0.0.1", 0))
            port = s.getsockname()[1]
        mp.start_processes(_worker, args=(port, world, name, most, median, str(tmp_path)), nprocs=world,
                           start_method="spawn")
        res[world] = np.load(tmp_path / f"g{world}.npz")
    for k in ("val", "err", "sums", "n", "rc", "evals", "iters"):
        assert np.array_equal(res[1][k], res[2][k]), k
