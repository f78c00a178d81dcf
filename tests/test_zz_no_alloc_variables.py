"""The allocation-free entry point on four and more inputs: its enclosures run on
shared-memory grids, where bern_propagate takes forms without a grid.  Collected with
test_zz_no_alloc.py, whose comparison and reasons for it hold here too."""
import numpy as np
import pytest

from test_zz_no_alloc import _close, _dev, _out
from paper_2211_14438_gb300 import bern
from paper_2211_14438_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("widths,cap", [
    ([4, 6, 6, 6, 1], 16),        # orders 1, 2, 4 and 8
    ([4, 6, 6, 6, 2], 7), ([4, 6, 6, 6, 1], 6), ([4, 6, 6, 1], 3), ([5, 5, 5, 1], 16),
    ([5, 5, 5, 5, 1], 5), ([6, 5, 5, 1], 16), ([6, 5, 5, 1], 3), ([7, 4, 1], 16), ([8, 3, 1], 16)])
def test_four_and_more_inputs(widths, cap):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    n, o, B = widths[0], widths[-1], 9
    net = wl.make_net(widths, 100 * n + cap)
    rng = np.random.default_rng(cap)
    c = rng.uniform(-1, 1, (B, n))
    boxes = np.stack([c - 0.3, c + 0.3], 2).astype(np.float32)
    W, b = _dev(net)
    bx = torch.from_numpy(boxes).cuda()
    terms = bern.max_output_terms(widths, 2, cap)
    ctx = bern.Context(0)
    want = ctx.propagate(widths, W, b, bx, degree=2, cap=cap, cap_terms=terms)
    want = {k: v for k, v in want.items() if v is not None}
    got = _out(B, o, terms)
    rc = bern.propagate_noalloc(widths, W, b, bx, got, degree=2, cap=cap)
    torch.cuda.synchronize()
    assert rc == bern.BERN_OK, bern.strerror(rc)
    _close(got, want)
    ctx.close()
