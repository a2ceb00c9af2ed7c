"""dfs_submit_new without a GPU: the plan of an expression, and refusals that
leave neither a task nor a store behind."""
import ctypes as C

import numpy as np
import pytest

from paper_2406_18109_gb300 import arrays as A
from paper_2406_18109_gb300 import binding as B
from tests.helpers import ensure_built


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def test_an_expression_is_the_same_plan():
    rt = A.Runtime(device=-1, tile=64)
    x, y = rt.empty((256,), np.float32), rt.empty((256,), np.float32)
    z = A.sqrt(x + 2.0 * y)                       # dfs_submit_new
    s = A.dot(z, z)
    plan = B.dfs_plan_json(rt.ctx)
    rt2 = A.Runtime(device=-1, tile=64)
    x, y = rt2.empty((256,), np.float32), rt2.empty((256,), np.float32)
    T, n = rt2.tiling((64,)), rt2.none
    t, u, z2 = (rt2.empty((256,), np.float32) for _ in range(3))
    s2 = rt2.empty((), np.float32)
    rt2.submit("MUL", (4,), [2.0, (y.handle, T, 1), (t.handle, T, 2)])
    rt2.submit("ADD", (4,), [(x.handle, T, 1), (t.handle, T, 1), (u.handle, T, 2)])
    rt2.submit("SQRT", (4,), [(u.handle, T, 1), (z2.handle, T, 2)])
    rt2.submit("DOT", (4,), [(z2.handle, T, 1), (z2.handle, T, 1), (s2.handle, n, 4)])
    t.release(), u.release()
    want = B.dfs_plan_json(rt2.ctx)
    assert [len(g) for g in plan["groups"]] == [len(g) for g in want["groups"]]
    assert len(plan["groups"]) == 1 and s.shape == () and z.shape == (256,)


@pytest.mark.parametrize("case", ["dtype", "op", "arity", "negative", "mixed"])
def test_refused(case):
    rt = A.Runtime(device=-1, tile=64)
    x = rt.empty((256,), np.float32)
    T = rt.tiling((64,))
    args = B.make_args([(x.handle, T, 1), (x.handle, T, 1), (x.handle, T, 2)])
    shape, dom, out = (C.c_int64 * 1)(256 if case != "negative" else -1), (C.c_int64 * 1)(4), C.c_int64(-5)
    before = rt.empty((8,), np.float32).handle
    rc = B.lib().dfs_submit_new(rt.ctx, 999 if case == "op" else 32, 1, dom, 9 if case == "arity" else 3, args,
                                7 if case == "dtype" else (1 if case == "mixed" else 0), 1, shape, C.byref(out))
    assert rc != 0 and out.value == -5 and B.dfs_last_error(rt.ctx)
    for h in range(before + 1, before + 4):       # nothing is left to view
        with pytest.raises(B.DfsError):
            B.dfs_store_view(rt.ctx, h, (0,), (1,))
    assert not B.dfs_plan_json(rt.ctx)["groups"]
