"""The variants of the enclosure where it runs on grids (two and three variables from
order 9 on, four and more from 10 on): every forced one gives the same bits."""
import numpy as np
import pytest

from test_gpu_enclose_orders import _graded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,l,D", [(1, 12, 12), (2, 9, 9), (2, 16, 16), (3, 9, 9), (3, 12, 10),
                                   (3, 16, 16), (4, 10, 10), (4, 11, 6)])
def test_variants_agree(n, l, D):
    import torch
    from paper_2211_14438_gb300 import bern
    B, h, M = 3, 7, len(_graded(n, D))
    rng = np.random.default_rng(100 * n + l)
    up = torch.from_numpy(rng.normal(size=(B, M, h)).astype(np.float32)).cuda()
    lo = up - 0.1
    nt = torch.from_numpy(rng.integers(1, M + 1, (B, h)).astype(np.int32)).cuda()
    ctx = bern.Context(0)
    got = []
    for v in range(5):
        ctx.force_variant("enclose", v)
        rl, ru = torch.zeros(B, h, device="cuda"), torch.zeros(B, h, device="cuda")
        ctx.enclose(n, B, h, l, 0, up, lo, M, nt, rl, ru)
        ctx.check("enclose")
        got.append((rl.cpu().numpy(), ru.cpu().numpy()))
    ctx.close()
    for rl, ru in got[1:]:
        assert np.array_equal(rl, got[0][0]) and np.array_equal(ru, got[0][1])
