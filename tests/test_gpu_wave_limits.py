"""The waits of in-place sweeps run out: CTA 0 withholds one flag (the test
hook), every wait ends at the time limit, the launch reports it, and the next
sweeps of the same context are right."""
import numpy as np
import pytest

from helpers import gpu_runtime
from paper_2406_18109_gb300 import binding as B
from test_gpu_waves import FIVE, SEVEN, _run, _sweep, _views

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape, offsets, per_flush, flag", [
    ((515, 700), FIVE, 1, 1),          # bands: edges read, first sweep
    ((515, 700), FIVE, 1, 3),          # ... second sweep (a launch of its own)
    ((515, 700), FIVE, 3, 5),          # ... third sweep of one launch
    ((40, 70, 81), SEVEN, 1, 1),       # tiles
    ((40, 70, 81), SEVEN, 3, 2),
], ids=str)
def test_a_withheld_flag_is_reported_and_the_context_survives(shape, offsets, per_flush, flag):
    host = np.random.default_rng(7).uniform(0.0, 1.0, shape).astype(np.float32)
    want, _ = _run("unfused", host, offsets, 4, 1, False)
    with gpu_runtime("persistent", timeout_s=0.05, debug_skip_arrival=-flag) as rt:
        views = _views(rt.array(host), offsets)
        # (with a grid barrier after the sweep, the CTAs already there may give up first)
        with pytest.raises(B.DfsError, match="in-place sweep timed out|grid barrier timed out" if flag == 2 else
                           "in-place sweep timed out") as e:
            for k in range(6):
                _sweep(views)
                if (k + 1) % per_flush == 0:
                    rt.wait(rt.record())
        assert e.value.code == -6
        assert "in-place sweep" in rt.kernel_source()
        rt.sync()                                # error consumed
        again = rt.array(host)                   # the numbers go on: no flag is withheld twice
        views = _views(again, offsets)
        for k in range(4):
            _sweep(views)
            if (k + 1) % 2 == 0:
                rt.flush()
        got = again.numpy()
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
