"""The sizing network on more rows than a grid's second dimension has blocks
(65535 blocks of 32 rows, GPU): prediction of the first and last rows against
the oracle at the network test's tolerance, and a training step."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2305_19768_gb300 import qmc

pytestmark = pytest.mark.gpu

ROWS = 65535 * 32 + 1


def test_more_than_two_million_rows():
    net = qmc.Mlp(2, 128, 1, 3, seed=7)
    try:
        rng = np.random.default_rng(5)
        x = rng.uniform(-1, 1, size=(ROWS, 2)).astype(np.float32)
        p = net.params()
        out = net.forward(x)
        for part in (slice(0, 256), slice(ROWS - 256, ROWS)):
            ref, _ = omlp.forward(p, x[part], 2, 128, 1, 3, bf16=True)
            assert np.abs(out[part] - ref).max() <= 5e-3 * np.abs(ref).max()
        y = np.sin(3 * x[:, :1] + np.arange(3, dtype=np.float32)).astype(np.float32)
        losses = net.train(x, y, 1, 1e-3)
        # the FP32 terms of the squared error, summed in FP64
        ref = float(((out.astype(np.float64) - y) ** 2).sum() / ROWS)
        assert abs(losses[0] - ref) <= 1e-5 * ref
        assert not np.array_equal(net.params(), p) and np.isfinite(net.params()).all()
    finally:
        net.close()
