"""Launch packing on the GPU: sweeps of the same arrays join although scalar
tasks stand between them, and only where nothing in between is used.  Every
result must be bit for bit what the unfused tasks give."""
import numpy as np
import pytest

from helpers import gpu_runtime
from paper_2406_18109_gb300 import arrays as A

pytestmark = pytest.mark.gpu


def _norms(rt, x, y):
    d = x - y
    nd = A.norm(d)
    s, p = A.asum(y), A.dot(x, y)
    return [d / nd, nd, s, p]


def _own_temporaries(rt, x, y):
    """The later sweep has temporaries, immediates and a result of its own."""
    a = A.norm(x)
    w = 2.0 * x + y
    b = A.asum(w * w)
    return [x / a, a, w, b]


def _uses_the_scalar(rt, x, y):
    """The later sweep reads what the scalar task made: it stays."""
    nd = A.norm(x)
    s = A.asum(x * nd)
    return [nd, s]


def _overwrites(rt, x, y):
    """The later sweep writes what the one between reads: order is kept."""
    nd = A.norm(x)
    z = y / nd
    y[...] = x
    return [nd, z, y, A.asum(y)]


@pytest.mark.parametrize("program, barriers", [(_norms, 1), (_own_temporaries, 1), (_uses_the_scalar, 1), (_overwrites, None)])
@pytest.mark.parametrize("n", [1, 3, 257, 4096, 70003, 1 << 20])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_packed_equals_unfused(program, barriers, n, dtype):
    r = np.random.default_rng(n)
    hx, hy = r.uniform(0.5, 1.0, n).astype(dtype), r.uniform(-1.0, 1.0, n).astype(dtype)
    outs = {}
    for mode in ("persistent", "unfused"):
        with gpu_runtime(mode) as rt:
            res = program(rt, rt.array(hx), rt.array(hy))
            rt.flush()
            if mode == "persistent" and barriers is not None and n > 4096:
                assert rt.kernel_source().count("grid_barrier(ctl") == barriers
            outs[mode] = [a.numpy() for a in res]
    for a, b in zip(outs["persistent"], outs["unfused"]):
        assert np.array_equal(np.atleast_1d(a).view(np.uint8), np.atleast_1d(b).view(np.uint8))


@pytest.mark.parametrize("offset", [0, 1, 3])
def test_sweeps_of_another_alignment_stay_apart(offset):
    """A sum over a view keeps its own order of addition."""
    h = np.random.default_rng(9).uniform(-1.0, 1.0, 100003).astype(np.float32)
    outs = {}
    for mode in ("persistent", "unfused"):
        with gpu_runtime(mode) as rt:
            x = rt.array(h)
            nd = A.norm(x)
            q = nd * 2.0
            s = A.asum(x[offset:])
            rt.flush()
            outs[mode] = [a.numpy() for a in (nd, q, s)]
    for a, b in zip(outs["persistent"], outs["unfused"]):
        assert np.atleast_1d(a).view(np.uint32) == np.atleast_1d(b).view(np.uint32)
