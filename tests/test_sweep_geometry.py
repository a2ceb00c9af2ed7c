"""Which form an in-place sweep takes, from the generated source (no GPU)."""
import numpy as np
import pytest

from paper_2406_18109_gb300 import arrays as A
from paper_2406_18109_gb300 import binding as B
from tests.helpers import ensure_built


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _source(program, **kw):
    """The kernel of the last launch of what program(rt) buffers; it compiles."""
    with A.Runtime(device=-1, **kw) as rt:
        keep = program(rt)  # noqa: F841
        with pytest.raises(B.DfsError, match="not launched"):
            rt.flush()
        return rt.kernel_source()


def _relax(g):
    c, n, e, w, s = g[1:-1, 1:-1], g[:-2, 1:-1], g[1:-1, 2:], g[1:-1, :-2], g[2:, 1:-1]
    work = 0.2 * (c + n + e + w + s)
    c[...] = work


@pytest.mark.parametrize("shape, rows, cols", [
    ((2 ** 31 + 10, 3), slice(None), slice(None)),                  # more rows than an int holds
    ((2 ** 31 - 1, 3), slice(None), slice(None)),                   # the last band's start would pass 2^31
    ((2 ** 33, 66), slice(2 ** 32, 2 ** 32 + 66), slice(None)),     # a small view far down
    ((66, 2 ** 33), slice(None), slice(2 ** 32, 2 ** 32 + 66)),     # and far along the rows
], ids=str)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_sides_beyond_32_bit_indices_take_two_phases(shape, rows, cols, dtype):
    src = _source(lambda rt: _relax(rt.empty(shape, dtype)[rows, cols]))
    assert "in-place sweep" not in src and "grid_barrier(ctl" in src


@pytest.mark.parametrize("shape, form", [((66, 66), " bands of "), ((2 ** 30 - 1, 3), " bands of "), ((65, 65), None)])
def test_ordinary_sides_are_swept_in_place(shape, form):
    src = _source(lambda rt: _relax(rt.empty(shape, np.float32)))
    assert (form in src) if form else "in-place sweep" not in src
