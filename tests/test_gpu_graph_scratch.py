"""Graphs replayed after the context's scratch has grown: the block that they
recorded stays theirs."""
import numpy as np
import pytest

from helpers import gpu_runtime
from paper_2406_18109_gb300 import arrays as A

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", [False, True])
def test_replay_after_the_scratch_has_grown(batched):
    r = np.random.default_rng(1)
    host = [r.uniform(-1.0, 1.0, n) for n in (5000, 20000, 70001)]
    with gpu_runtime("persistent", tile=256) as rt:
        xs = [rt.array(h) for h in host]
        ss = [rt.scalar(0.0, np.float64) for _ in host]

        def step():
            if batched:
                rt.batch_begin()
            for x, s in zip(xs, ss):
                s[...] = A.dot(x, x)
                if batched:
                    rt.batch_next()
            rt.batch_end() if batched else rt.flush()

        step()
        want = [s.item() for s in ss]
        rt.capture_begin()
        step()
        graph = rt.capture_end()
        big = rt.array(np.ones(1 << 26, dtype=np.float32))      # 262144 points: two megabytes of partials
        many = [rt.array(np.full(300, float(i))) for i in range(400)]
        for _ in range(2):
            total = A.asum(big)
            rt.flush()
            rt.batch_begin()                                    # more batch scalars
            for v in many:
                v *= A.dot(v, v) * 0.0 + 1.0
                rt.batch_next()
            rt.batch_end()
            rt.sync()
            filler = rt.array(np.full(1 << 18, np.nan))         # takes what was given back
            for s in ss:
                s[...] = 0.0
            rt.graph_launch(graph)
            assert [s.item() for s in ss] == want
            assert total.item() == float(1 << 26)
            del filler
        rt.graph_destroy(graph)
        step()
        assert [s.item() for s in ss] == want
