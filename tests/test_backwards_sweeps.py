"""Which flat sweeps run from the end (no GPU)."""
import numpy as np
import pytest

from paper_2406_18109_gb300 import arrays as A
from paper_2406_18109_gb300 import binding as B
from tests.helpers import ensure_built


@pytest.mark.parametrize("n, dtype, backwards", [(1 << 24, np.float32, True), (1 << 24, np.float64, False), (1 << 21, np.float64, True)])
def test_fp64_sweeps_beyond_l2_run_from_the_start(n, dtype, backwards):
    ensure_built()
    with A.Runtime(device=-1) as rt:
        x, y = rt.empty((n,), dtype), rt.empty((n,), dtype)
        s = A.asum(x) * 2.0
        out = [y * 3.0, x + s]  # noqa: F841
        with pytest.raises(B.DfsError, match="not launched"):
            rt.flush()
        src = rt.kernel_source()
    assert ("nv - 1 - (" in src) == backwards
