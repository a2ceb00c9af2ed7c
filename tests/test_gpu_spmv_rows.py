"""FP32 row products a warp's rows at a time (spmv_rows): empty rows, rows
longer than a chunk, ragged ends, decreasing row bounds, alone and batched."""
import numpy as np
import pytest

from helpers import gpu_runtime
from paper_2406_18109_gb300 import arrays as A

pytestmark = pytest.mark.gpu


def _matrix(lengths, ncols, seed):
    r = np.random.default_rng(seed)
    rp = np.zeros(len(lengths) + 1, dtype=np.int32)
    rp[1:] = np.cumsum(lengths)
    col = r.integers(0, ncols, rp[-1]).astype(np.int32)
    return rp, col, r.uniform(-1.0, 1.0, rp[-1]).astype(np.float32)


def _check(rp, col, val, x, y):
    """|y - A x| <= (row length + 1) eps |A| |x|, the bound of a sum of fused
    multiply-adds in any order."""
    for i in range(len(rp) - 1):
        k = slice(rp[i], max(rp[i], rp[i + 1]))
        p = val[k].astype(np.float64) * x[col[k]].astype(np.float64)
        assert abs(float(y[i]) - p.sum()) <= (len(p) + 1) * 2.0 ** -24 * np.abs(p).sum(), i


CASES = {
    "empty": [0] * 300,
    "one row": [5],
    "ragged": list(np.random.default_rng(1).integers(0, 40, 517)),
    "five": [5] * 1025,
    "chunk edges": [8] * 31 + [128, 127, 1, 0, 256, 255, 257] + [3] * 90,
    "long rows": [1] * 400 + [5000, 0, 3, 1200] + [2] * 700,
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("kw", [dict(), dict(tile=256, block=128), dict(tile=128, block=1024, unroll=1)], ids=str)
def test_rows(name, kw):
    lengths = CASES[name]
    x = np.random.default_rng(2).uniform(-1.0, 1.0, 900).astype(np.float32)
    rp, col, val = _matrix(lengths, len(x), 3)
    got = {}
    for mode in ("persistent", "unfused"):
        with gpu_runtime(mode, **kw) as rt:
            Am = A.CSR(rt, rp, col, val, ncols=len(x)) if len(x) != len(lengths) else A.CSR(rt, rp, col, val)
            y = Am @ rt.array(x)
            s = A.dot(y, y)
            rt.flush()
            if mode == "persistent":
                assert "spmv_rows<float" in rt.kernel_source()
            got[mode] = (y.numpy(), s.numpy())
    _check(rp, col, val, x, got["persistent"][0])
    for a, b in zip(got["persistent"], got["unfused"]):
        assert np.array_equal(np.atleast_1d(a).view(np.uint32), np.atleast_1d(b).view(np.uint32))


def test_decreasing_row_bounds():
    """Not a CSR matrix, but accepted: rows end before they begin (empty), and
    later rows read entries again."""
    r = np.random.default_rng(5)
    rp = np.array([0, 7, 3, 12, 12, 5, 40] + [40 + 2 * (i % 3) for i in range(200)], dtype=np.int32)
    rp[-1] = 60
    col = r.integers(0, 50, 60).astype(np.int32)
    val = r.uniform(-1.0, 1.0, 60).astype(np.float32)
    x = r.uniform(-1.0, 1.0, 50).astype(np.float32)
    with gpu_runtime("persistent") as rt:
        y = (A.CSR(rt, rp, col, val, ncols=50) @ rt.array(x)).numpy()
    _check(rp, col, val, x, y)


def test_batched_rows_equal_alone():
    """Solves of different row lengths (dealt longest first) in one launch."""
    probs = [_matrix(np.random.default_rng(s).integers(lo, hi, n), n, s)
             for s, (lo, hi, n) in enumerate([(1, 9, 700), (8, 40, 3001), (5, 6, 5000), (0, 3, 1030)])]
    xs = [np.random.default_rng(10 + i).uniform(-1.0, 1.0, len(p[0]) - 1).astype(np.float32) for i, p in enumerate(probs)]
    outs = {}
    for mode in ("alone", "batched"):
        with gpu_runtime("persistent", tile=512) as rt:
            state = [(A.CSR(rt, *p), rt.array(x), rt.array(np.zeros_like(x)), rt.scalar(0.0, np.float32))
                     for p, x in zip(probs, xs)]
            rt.flush()
            if mode == "batched":
                rt.batch_begin()
            for Am, x, y, s in state:
                Am.spmv(x, y)
                s[...] = A.dot(x, y)
                rt.batch_next() if mode == "batched" else rt.flush()
            if mode == "batched":
                rt.batch_end()
                assert rt.stats()["batch_fallbacks"] == 0 and "spmv_rows<float" in rt.kernel_source()
            outs[mode] = [(y.numpy(), s.numpy()) for _, _, y, s in state]
    for a, b in zip(outs["alone"], outs["batched"]):
        assert np.array_equal(a[0].view(np.uint32), b[0].view(np.uint32)) and a[1] == b[1]
