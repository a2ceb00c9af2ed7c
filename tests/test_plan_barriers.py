"""dfs_plan_json's barriers are those of the kernel that is launched (no GPU)."""
import numpy as np
import pytest

from paper_2406_18109_gb300 import arrays as A
from paper_2406_18109_gb300 import binding as B
from paper_2406_18109_gb300 import workloads as W
from tests.helpers import ensure_built


def _sweep(rt):
    views = W.jacobi_views(rt.empty((200, 300), np.float32))
    W.jacobi_sweep(views)
    return views


def _sweep_and_norms(rt):
    v, x = _sweep(rt), rt.empty((100000,), np.float32)
    n = A.norm(x)
    return v, n, A.asum(x) * n, x / n


def _norms(rt):
    x, y = rt.empty((100000,), np.float64), rt.empty((100000,), np.float64)
    n = A.norm(x)
    q = A.asum(x) * 2.0                           # joins the sum of squares
    return n, q, A.dot(x, y), y / q


def _small_sweep(rt):
    views = W.jacobi_views(rt.empty((20, 30), np.float32))
    W.jacobi_sweep(views)
    return views


@pytest.mark.parametrize("program, fewer", [(_sweep, True), (_sweep_and_norms, True), (_norms, True), (_small_sweep, False)])
def test_barriers_of_the_plan(program, fewer):
    ensure_built()
    with A.Runtime(device=-1) as rt:
        keep = program(rt)  # noqa: F841
        p = rt.plan()
        scalar = set(p["scalar_groups"])
        cuts = sum(1 for groups in p["launches"] for g in groups[:-1] if g not in scalar)
        with pytest.raises(B.DfsError, match="not launched"):
            rt.flush()
        src = rt.kernel_source()
    assert p["barriers"] == src.count("grid_barrier(ctl")
    assert (p["barriers"] < cuts) if fewer else (p["barriers"] == cuts)
