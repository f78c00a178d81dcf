"""Enclosures at orders below the degree: the terms above the order are added by
all threads of a block, in as many parts as its items leave threads.  One item to
several blocks of them, ragged counts around the order's last term."""
import numpy as np
import pytest

from test_gpu_enclose_orders import _graded, _range

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,l,D,B,h", [
    (1, 4, 16, 3, 50), (2, 2, 16, 1, 1), (2, 2, 16, 40, 33), (2, 8, 16, 2, 9), (2, 5, 9, 700, 64),
    (3, 2, 16, 1, 1), (3, 2, 9, 300, 40), (3, 8, 13, 2, 15), (4, 2, 8, 1, 45), (4, 4, 8, 2, 3),
    (4, 6, 8, 1, 5), (5, 2, 6, 2, 9), (6, 2, 8, 1, 3), (6, 3, 8, 1, 2), (7, 2, 6, 1, 3),
    (8, 2, 5, 1, 3), (8, 3, 5, 1, 2), (1, 1, 16, 2, 5), (3, 1, 12, 1, 1), (3, 1, 12, 900, 64),
    (6, 1, 8, 1, 3), (8, 1, 6, 2, 3), (2, 1, 16, 20, 33)])
def test_orders_below_the_degree(n, l, D, B, h):
    import torch
    from paper_2211_14438_gb300 import bern
    rng = np.random.default_rng(1000 * n + 10 * l + D)
    e = _graded(n, D)
    M, own = len(e), len(_graded(n, l))
    up = rng.normal(size=(B, M, h)).astype(np.float32)
    lo = rng.normal(size=(B, M, h)).astype(np.float32)
    nt = rng.choice([own - 1, own, own + 1, (own + M) // 2, M - 1, M], (B, h)).astype(np.int32)
    nt[0, 0] = M
    dev = [torch.from_numpy(x).cuda() for x in (up, lo, nt)]
    rl, ru = torch.zeros(B, h, device="cuda"), torch.zeros(B, h, device="cuda")
    ctx = bern.Context(0)
    ctx.enclose(n, B, h, l, 0, dev[0], dev[1], M, dev[2], rl, ru)
    ctx.check("enclose")
    ctx.close()
    rl, ru = rl.cpu().numpy().astype(np.float64), ru.cpu().numpy().astype(np.float64)
    flat = rng.permutation(B * h)[:20]
    flat[0] = 0
    for b, m in zip(flat // h, flat % h):
        k = nt[b, m]
        au, al = up[b, :k, m].astype(np.float64), lo[b, :k, m].astype(np.float64)
        hi, lw = _range(n, l, e[:k], au)[1], _range(n, l, e[:k], al)[0]
        # every coefficient is a sum with weights in [0, 1]; a pass adds at most l
        # roundings of 2^-23, the scaling two, the terms above the order one each
        tol = (n * l + M + 4) * 2.0 ** -23
        assert hi - 1e-12 <= ru[b, m] <= hi + tol * np.abs(au).sum(), (b, m)
        assert lw + 1e-12 >= rl[b, m] >= lw - tol * np.abs(al).sum(), (b, m)
