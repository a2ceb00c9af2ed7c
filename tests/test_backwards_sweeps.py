"""Which flat sweeps run from the end (no GPU)."""
import numpy as np
import pytest

from paper_2406_18109_gb300 import arrays as A
from paper_2406_18109_gb300 import binding as B
from tests.helpers import ensure_built


@pytest.mark.parametrize("dtype, backwards", [(np.float32, True), (np.float64, False)])
def test_only_fp32_sweeps_run_from_the_end(dtype, backwards):
    ensure_built()
    with A.Runtime(device=-1) as rt:
        x, y = rt.empty((1 << 24,), dtype), rt.empty((1 << 24,), dtype)
        s = A.asum(x) * 2.0
        out = [y * 3.0, x + s]  # noqa: F841
        with pytest.raises(B.DfsError, match="not launched"):
            rt.flush()
        src = rt.kernel_source()
    assert ("nv - 1 - (" in src) == backwards
