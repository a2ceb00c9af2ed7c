"""In-place sweeps on the GPU: a pair of groups that the anti-dependence
constraint cuts (a stencil over shifted views, then the copy into the centre)
runs as one sweep that never stores the intermediate result.  Every grid must
come out bit for bit as the unfused tasks leave it."""
import numpy as np
import pytest

from helpers import gpu_runtime
from paper_2406_18109_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FIVE = ((0, 0), (-1, 0), (0, 1), (0, -1), (1, 0))
SEVEN = ((0, 0, 0), (-1, 0, 0), (1, 0, 0), (0, -1, 0), (0, 1, 0), (0, 0, -1), (0, 0, 1))


def _views(g, offsets):
    """Shifted views of g, the written one (no offset) first."""
    nd = len(offsets[0])
    lo = [max(0, -min(o[d] for o in offsets)) for d in range(nd)]
    hi = [g.shape[d] - max(0, max(o[d] for o in offsets)) for d in range(nd)]
    return [g[tuple(slice(lo[d] + o[d], hi[d] + o[d]) for d in range(nd))] for o in offsets]


def _sweep(views):
    acc = views[0]
    for v in views[1:]:
        acc = acc + v
    work = (1.0 / len(views)) * acc
    views[0][...] = work


def _run(mode, host, offsets, sweeps, per_flush, wrap, **kw):
    with gpu_runtime(mode, **kw) as rt:
        if wrap:
            import torch
            g = rt.wrap(torch.from_numpy(host).cuda())
        else:
            g = rt.array(host)
        views = _views(g, offsets)
        for k in range(sweeps):
            _sweep(views)
            if (k + 1) % per_flush == 0:
                rt.flush()
        out = g.numpy()
        src = rt.kernel_source()
    return out, "in-place sweep" in src


def _check(shape, dtype, offsets, kw, wave=True):
    host = np.random.default_rng(3).uniform(0.0, 1.0, shape).astype(dtype)
    want, _ = _run("unfused", host, offsets, 3, 1, False, **kw)
    for per_flush, wrap in ((1, False), (3, False), (3, True)):
        got, w = _run("persistent", host, offsets, 3, per_flush, wrap, **kw)
        assert np.array_equal(got.view(np.uint8), want.view(np.uint8)), (per_flush, wrap)
        if not wrap and wave is not None:
            assert w == wave


@pytest.mark.parametrize("shape", [(66, 66), (64, 67), (131, 129), (257, 1023), (1021, 1147), (5000, 5), (900, 23), (5, 5000),
                                   (42, 9003), (19, 33003), (70, 64)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("kw", [dict(), dict(block=128), dict(block=1024, unroll=1), dict(ctas_per_sm=2)])
def test_2d_sweeps_equal_unfused(shape, dtype, kw):
    """Bands of one row and of many, several bands per CTA, panels, ragged
    edges; pitched rows (vectors) and dense ones (elements)."""
    _check(shape, dtype, FIVE, kw, wave=None if shape[1] > 9000 else bool((shape[0] - 2) * (shape[1] - 2) >= 4096))


@pytest.mark.parametrize("shape", [(18, 17, 21), (19, 130, 35), (40, 64, 66), (5, 300, 301)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("kw", [dict(), dict(block=128), dict(block=1024, unroll=1)])
def test_3d_sweeps_equal_unfused(shape, dtype, kw):
    """Tile edges, ragged last slices, more tiles than CTAs and fewer."""
    _check(shape, dtype, SEVEN, kw, wave=None)


@pytest.mark.parametrize("offsets", [
    ((0, 0), (1, 0)), ((0, 0), (-1, 0)), ((0, 0), (0, 1)), ((0, 0), (0, -1)),   # one-sided: the view touches the edge
    ((0, 0), (-1, -1), (-1, 1), (1, -1), (1, 1)),                                # diagonals
    ((0, 0), (0, 2), (0, -3)), ((0, 0), (0, 5)),                                 # further along the row
    ((0, 0), (2, 0), (0, 1)), ((0, 0), (-3, 2)),                                 # further rows (tiles, not bands)
], ids=str)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_other_stencils_equal_unfused(offsets, dtype):
    _check((203, 517), dtype, offsets, {}, wave=None)


def test_sweep_with_a_live_intermediate():
    """The application keeps `work`: it is stored as well as the centre."""
    host = np.random.default_rng(4).uniform(0.0, 1.0, (200, 333)).astype(np.float32)
    outs = {}
    for mode in ("persistent", "unfused"):
        with gpu_runtime(mode) as rt:
            g = rt.array(host)
            c, n, e, w, s = W.jacobi_views(g)
            work = 0.2 * (c + n + e + w + s)
            c[:] = work
            outs[mode] = (g.numpy(), work.numpy())
    for a, b in zip(outs["persistent"], outs["unfused"]):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))


@pytest.mark.parametrize("offsets, shape", [(FIVE, (515, 700)), (SEVEN, (40, 70, 81))])
def test_sweeps_replayed_from_a_graph(offsets, shape):
    """Captured sweeps (flags are numbered across launches, never cleared)."""
    host = np.random.default_rng(5).uniform(0.0, 1.0, shape).astype(np.float32)
    want, _ = _run("unfused", host, offsets, 12, 1, False)
    with gpu_runtime("persistent") as rt:
        g = rt.array(host)
        views = _views(g, offsets)
        rt.capture_begin()                 # first use of a sweep inside a capture
        for _ in range(2):
            _sweep(views)
            rt.flush()
        graph = rt.capture_end()
        for _ in range(6):
            rt.graph_launch(graph)
        got = g.numpy()
        rt.graph_destroy(graph)
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("shape, offsets", [((515, 700), FIVE), ((40, 70, 81), SEVEN)], ids=["2d", "3d"])
@pytest.mark.parametrize("kw", [dict(ctas_per_sm=8), dict(ctas_per_sm=4, block=1024), dict(ctas_per_sm=16, block=128)], ids=str)
def test_sweeps_with_more_ctas_asked_than_fit(shape, offsets, kw):
    """A ctas_per_sm that the sweep's kernel cannot reach: two phases then."""
    _check(shape, np.float32, offsets, kw, wave=None)


def test_sweeps_around_a_batch_that_grows_its_scratch():
    """A batch reallocates its own scratch only: the sweeps' flags stay."""
    from paper_2406_18109_gb300 import arrays as A
    host = np.random.default_rng(6).uniform(0.0, 1.0, (203, 517)).astype(np.float32)
    want, _ = _run("unfused", host, FIVE, 6, 1, False)
    with gpu_runtime("persistent") as rt:
        g = rt.array(host)
        views = _views(g, FIVE)
        for count in (1, 3, 40):
            for _ in range(2):
                _sweep(views)
                rt.flush()
            vs = [rt.array(np.full(3000, i, dtype=np.float32)) for i in range(count)]
            rt.batch_begin()
            for v in vs:
                v *= A.dot(v, v)
                rt.batch_next()
            rt.batch_end()
        got = g.numpy()
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
