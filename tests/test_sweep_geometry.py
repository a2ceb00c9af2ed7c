"""Which form an in-place sweep takes, from the generated source (no GPU)."""
import random
import re

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


@pytest.mark.parametrize("shape, form", [((66, 66), " bands of "), ((2 ** 30 - 1, 3000), " bands of "), ((65, 65), None)])
def test_ordinary_sides_are_swept_in_place(shape, form):
    src = _source(lambda rt: _relax(rt.empty(shape, np.float32)))
    assert (form in src) if form else "in-place sweep" not in src


def _relax_and_keep(rt, shape, dtype, negated):
    """The application keeps the intermediate, in views of the centre's phase."""
    inside = tuple(slice(1, -1) for _ in shape)
    g, kept = rt.empty(shape, dtype), rt.empty(shape, dtype)[inside]
    acc = g[inside]
    for d in range(len(shape)):
        for o in (slice(0, -2), slice(2, None)):
            acc = acc + g[tuple(o if k == d else slice(1, -1) for k in range(len(shape)))]
    kept[...] = 0.125 * acc
    g[inside][...] = -kept if negated else kept
    return g, kept


@pytest.mark.parametrize("shape", [(200, 333), (200, 336), (34, 34, 35)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("negated", [False, True])
def test_the_word_of_the_values_read_does_not_cancel(shape, dtype, negated):
    """A tile's arrival waits for a word made of all its results: it must depend
    on them where the sweep stores one value twice, or a value and its negation."""
    src = _source(lambda rt: _relax_and_keep(rt, shape, dtype, negated))
    assert "in-place sweep of" in src and " bands of " not in src
    lines = re.findall(r"u32 used_ = ([^;]*);|\n +used_ = ([^;]*);", src)
    arg = re.search(r"wave_read_done\(&wsync_, wrd_ \+ \(live \? 1u : 0u\), (.*)\);", src).group(1)
    names = re.findall(r"bits_of\((n\d+)(_[^)]*)\)", arg + "".join(a + b for a, b in lines))
    assert {n for n, _ in names} == {"n0", "n1"}

    def word(vals):
        def ev(expr, used):
            expr = re.sub(r"bits_of\(n(\d+)(_[^)]*)\)",
                          lambda m: str(vals[m.group(2)] ^ (0x80000000 if negated and m.group(1) == "1" else 0)), expr)
            rotl = lambda a, b, k: (a << k | b >> (32 - k)) & 0xffffffff  # noqa: E731
            return eval(re.sub(r"\b(\d+)u\b", r"\1", expr), {"used_": used, "__funnelshift_l": rotl}) & 0xffffffff
        used = None
        for a, b in lines:
            used = ev(a or b, used)
        return ev(arg, used)

    r = random.Random(1)
    elems = {e for _, e in names}
    assert len({word({e: r.getrandbits(32) for e in elems}) for _ in range(16)}) == 16


@pytest.mark.parametrize("shape, kw", [((17400, 10400), {}), ((43000, 4104), dict(block=1024, unroll=1)),
                                       ((30000, 8232), dict(block=512))], ids=str)
def test_edge_columns_of_a_panel_are_read_whole(shape, kw):
    """Rows of several panels: the columns next to a panel, all rows of a band,
    are read by the threads that own vectors (fewer than the CTA's)."""
    src = _source(lambda rt: _relax(rt.empty(shape, np.float32)), **kw)
    rows, = re.findall(r" bands of (\d+) rows", src)
    own, = set(re.findall(r"grp < 1 && q < (\d+)", src))
    loops = set(re.findall(r"i < rz - ra \+ 2; i \+= (\d+)\)", src))
    assert len(loops) == 1
    seen = {i for q in range(int(own)) for i in range(q, int(rows) + 2, int(*loops))}
    assert seen == set(range(int(rows) + 2))


def _seven(g):
    c = g[1:-1, 1:-1, 1:-1]
    acc = c + g[:-2, 1:-1, 1:-1] + g[2:, 1:-1, 1:-1] + g[1:-1, :-2, 1:-1] + g[1:-1, 2:, 1:-1] + g[1:-1, 1:-1, :-2] + g[1:-1, 1:-1, 2:]
    work = (1.0 / 7) * acc
    c[...] = work


@pytest.mark.parametrize("program, shape, dtype, form", [
    # narrow rows leave most lanes of a band idle
    ("relax", (1000002, 5), np.float32, None), ("relax", (1000002, 5), np.float64, None),
    ("relax", (200002, 34), np.float32, None), ("relax", (200002, 34), np.float64, None),
    # a second result in memory, FP32
    ("keep", (2050, 2050), np.float32, None), ("keep", (200, 200, 200), np.float32, None),
    # readers nearly a round away; short rows that waste lanes, FP64
    ("seven", (22, 502, 502), np.float64, None), ("seven", (502, 502, 22), np.float64, None),
    # where they are faster: bands (with several groups of warps, with panels), tiles
    ("relax", (8192, 8192), np.float32, " bands of "), ("relax", (20002, 302), np.float32, " bands of "),
    ("relax", (302, 20002), np.float32, " bands of "), ("relax", (1023, 1149), np.float64, " bands of "),
    ("seven", (253, 253, 253), np.float32, " tiles"), ("seven", (253, 253, 253), np.float64, " tiles"),
], ids=str)
def test_sweeps_are_in_place_where_that_is_faster(program, shape, dtype, form):
    src = _source(lambda rt: _relax_and_keep(rt, shape, dtype, False) if program == "keep"
                  else (_relax if program == "relax" else _seven)(rt.empty(shape, dtype)))
    assert ("in-place sweep" in src and form in src) if form else "in-place sweep" not in src
