"""Bands of several groups of warps in a CTA, with one and more vectors per
thread: every grid as the unfused tasks leave it, bit for bit."""
import re

import numpy as np
import pytest

from helpers import gpu_runtime
from test_gpu_waves import FIVE, _run, _sweep, _views

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(300, 300), (514, 514), (700, 700), (1026, 1026), (3000, 130), (2000, 1201)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("kw", [dict(), dict(block=512)], ids=str)
def test_groups_equal_unfused(shape, dtype, kw):
    host = np.random.default_rng(11).uniform(0.0, 1.0, shape).astype(dtype)
    want, _ = _run("unfused", host, FIVE, 4, 1, False, **kw)
    with gpu_runtime("persistent", **kw) as rt:
        views = _views(rt.array(host), FIVE)
        for k in range(4):
            _sweep(views)
            if k != 1:                        # launches of one sweep and of two
                rt.flush()
        src = rt.kernel_source()
        out = host.copy()
        out[1:-1, 1:-1] = views[0].numpy()
    assert np.array_equal(out.view(np.uint8), want.view(np.uint8))
    if dtype == np.float32:
        assert re.search(r" bands of ", src)
