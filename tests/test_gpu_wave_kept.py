"""In-place sweeps that store two results: the application keeps the
intermediate, in views of the centre's column phase."""
import numpy as np
import pytest

from helpers import gpu_runtime
from test_gpu_waves import FIVE, SEVEN, _views

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(200, 333), (200, 336), (34, 34, 35)], ids=str)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("negated", [False, True])
@pytest.mark.parametrize("per_flush", [1, 3])
def test_two_results_equal_unfused(shape, dtype, negated, per_flush):
    offsets = FIVE if len(shape) == 2 else SEVEN
    host = np.random.default_rng(12).uniform(0.0, 1.0, shape).astype(dtype)
    outs = {}
    for mode in ("persistent", "unfused"):
        with gpu_runtime(mode) as rt:
            g, k = rt.array(host), rt.array(np.zeros_like(host))
            views, kept = _views(g, offsets), _views(k, offsets)[0]
            for i in range(6):
                acc = views[0]
                for v in views[1:]:
                    acc = acc + v
                kept[...] = (1.0 / len(views)) * acc
                views[0][...] = -kept if negated else kept
                del acc
                if (i + 1) % per_flush == 0:
                    rt.flush()
            if mode == "persistent":
                src = rt.kernel_source()
                assert "in-place sweep of" in src and " bands of " not in src
            outs[mode] = (g.numpy(), k.numpy())
    for a, b in zip(outs["persistent"], outs["unfused"]):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
