"""Joined FP64 sweeps that would need a second round of points stay apart."""
import numpy as np
import pytest

from helpers import gpu_runtime
from paper_2406_18109_gb300 import arrays as A

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_points_in_one_round(dtype):
    n = 4000000                                   # 601 points of 6656 elements over 608 CTAs of 64 registers
    r = np.random.default_rng(1)
    hx, hy = r.uniform(0.5, 1.0, n).astype(dtype), r.uniform(0.5, 1.0, n).astype(dtype)
    outs = {}
    for mode in ("persistent", "unfused"):
        with gpu_runtime(mode) as rt:
            x, y, z = rt.array(hx), rt.array(hy), rt.array(np.zeros_like(hx))
            q, u = rt.scalar(0.0, dtype), rt.scalar(0.0, dtype)
            rt.flush()
            nd = A.norm(x)
            z[...] = x / nd
            q[...] = A.asum(y)
            u[...] = A.dot(x, y)
            rt.flush()
            if mode == "persistent":
                points = rt.layout((n,))[0][0]
                assert points <= 608 and rt.stats()["last_grid"] >= points
            outs[mode] = [a.numpy() for a in (z, q, u)]
    for a, b in zip(outs["persistent"], outs["unfused"]):
        assert np.array_equal(np.atleast_1d(a).view(np.uint8), np.atleast_1d(b).view(np.uint8))
