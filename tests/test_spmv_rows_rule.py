"""Which FP32 SpMVs are computed a warp's rows at a time (no GPU)."""
import numpy as np
import pytest

from paper_2406_18109_gb300 import arrays as A
from paper_2406_18109_gb300 import binding as B
from tests.helpers import ensure_built


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _source(rows, nnz, dtype, **kw):
    with A.Runtime(device=-1, **kw) as rt:
        Am = A.CSR.__new__(A.CSR)
        Am.rt, Am.nrows, Am.ncols, Am.nnz, Am.dtype = rt, rows, rows, nnz, np.dtype(dtype)
        Am.rowptr, Am.col, Am.val = rt.empty((rows + 1,), np.int32), rt.empty((nnz,), np.int32), rt.empty((nnz,), dtype)
        x, y = rt.empty((rows,), dtype), rt.empty((rows,), dtype)
        Am.spmv(x, y)
        with pytest.raises(B.DfsError, match="not launched"):
            rt.flush()
        return rt.kernel_source()


@pytest.mark.parametrize("rows, entries, kw, by_rows", [
    (1000000, 5, {}, True), (1000000, 31, {}, True), (100000, 31, {}, True), (10000, 5, {}, True), (1000, 16, {}, True),
    (4000000, 1, {}, False), (1000000, 1, {}, True),
    (1000, 31, {}, False), (40000, 31, {}, False),
    (100000, 5, dict(block=512), False), (100000, 31, dict(block=512), False), (1000000, 5, dict(block=512), True),
    (100000, 16, dict(block=1024), False), (1000000, 5, dict(block=1024), False), (1000000, 16, dict(block=1024), True),
], ids=str)
def test_rule(rows, entries, kw, by_rows):
    src = _source(rows, rows * entries, np.float32, **kw)
    assert ("spmv_rows<float" in src) == by_rows and ("spmv_row<float>" in src) != by_rows
    assert "spmv_rows<" not in _source(rows, rows * entries, np.float64, **kw)
