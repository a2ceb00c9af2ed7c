"""Bands of many rows in panels narrower than the CTA: the columns next to a
panel must be there for every row of the band."""
import pytest

from helpers import gpu_runtime
from test_gpu_waves import FIVE, _sweep, _views

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape, kw", [((17400, 10400), {}), ((43000, 4104), dict(block=1024, unroll=1))], ids=str)
def test_tall_panels_equal_unfused(shape, kw):
    torch = pytest.importorskip("torch")
    g = torch.rand(shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(8))
    outs = []
    for mode in ("persistent", "unfused"):
        x = g.clone()
        torch.cuda.synchronize()
        with gpu_runtime(mode, **kw) as rt:
            views = _views(rt.wrap(x), FIVE)
            for _ in range(2):
                _sweep(views)
                rt.flush()
            rt.sync()
            if mode == "persistent":
                assert "panel(s)" in rt.kernel_source() and ", 1 panel(s)" not in rt.kernel_source()
        outs.append(x)
    assert torch.equal(outs[0].view(torch.int32), outs[1].view(torch.int32))
