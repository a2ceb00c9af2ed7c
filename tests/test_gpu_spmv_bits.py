"""The bits of FP32 row products: fused multiply-adds in entry order, from the
host's exact arithmetic (rows longer than a chunk of spmv_rows, empty rows)."""
from fractions import Fraction

import numpy as np
import pytest

from helpers import gpu_runtime
from paper_2406_18109_gb300 import arrays as A
from test_gpu_spmv_rows import CASES, _matrix

pytestmark = pytest.mark.gpu


def _round32(q):
    """The FP32 value nearest to an exact rational, ties to even."""
    d = float(q)                                  # nearest double
    lo = np.float32(d)
    if float(lo) == d:
        return lo if Fraction(d) == q else np.float32(d)   # d is an FP32 value: within half an ulp of q
    hi = np.nextafter(lo, np.float32(np.inf if float(lo) < d else -np.inf))
    if 2 * Fraction(d) != Fraction(float(lo)) + Fraction(float(hi)) or Fraction(d) == q:
        return lo                                 # no tie, or a true one (the conversion broke it to even)
    return max(lo, hi) if q > Fraction(d) else min(lo, hi)


def _row(val, x):
    acc = np.float32(0.0)
    for v, w in zip(val, x):
        acc = _round32(Fraction(float(v)) * Fraction(float(w)) + Fraction(float(acc)))
    return acc


@pytest.mark.parametrize("name", CASES)
def test_rows_are_fused_multiply_adds_in_order(name):
    x = np.random.default_rng(2).uniform(-1.0, 1.0, 900).astype(np.float32)
    rp, col, val = _matrix(CASES[name], len(x), 3)
    with gpu_runtime("persistent") as rt:
        y = (A.CSR(rt, rp, col, val, ncols=len(x)) @ rt.array(x)).numpy()
        assert "spmv_rows<float" in rt.kernel_source()
    want = np.array([_row(val[a:b], x[col[a:b]]) for a, b in zip(rp[:-1], rp[1:])], dtype=np.float32)
    assert np.array_equal(y.view(np.uint32), want.view(np.uint32))
