"""Squares of short and medium inputs (up to 50 padded terms): whether a warp, two or a
block take a group depends on the neurons of the call, and changes nothing."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,D,B,h,share", [
    (2, 7, 1100, 64, 1.0), (2, 8, 1100, 64, 1.0), (2, 8, 2600, 60, 0.3), (2, 8, 1101, 63, 0.5),
    (3, 4, 1100, 64, 1.0), (3, 4, 1101, 63, 0.01), (2, 3, 700, 64, 1.0), (1, 1, 701, 63, 0.6),
    (1, 8, 1400, 64, 1.0)])
@pytest.mark.parametrize("place", [False, True])
def test_forms_of_medium_squares(n, D, B, h, share, place):
    import torch
    from paper_2211_14438_gb300 import bern
    g = torch.Generator(device="cuda").manual_seed(100 * n + D)
    M, keep = bern.num_monomials(n, D), bern.num_monomials(n, 2 * D)
    rnd = lambda *s: torch.rand(*s, device="cuda", generator=g)
    up, lo = rnd(B, M, h) - 0.4, rnd(B, M, h) - 0.6
    nt = torch.full((B, h), M, dtype=torch.int32, device="cuda")
    nt[:, ::3] = bern.num_monomials(n, D - 1)          # a lower degree
    L, H = -1.0 - rnd(B, h), 1.0 + rnd(B, h)
    kind = torch.where(rnd(B, h) < share, 2, 1).to(torch.int8)
    coef, eps = rnd(B, h, bern.COEF_STRIDE), rnd(B, h)
    ctx = bern.Context(0)

    def run(b0, b1):
        pn = torch.zeros(b1 - b0, h, dtype=torch.int32, device="cuda")
        pu, pl = (torch.zeros(b1 - b0, keep, h, device="cuda") for _ in range(2))
        src, ld = (up[b0:b1].contiguous(), lo[b0:b1].contiguous()), M
        if place:
            pu[:, :M], pl[:, :M] = src
            src, ld = (pu, pl), keep
        ctx.compose(n, b1 - b0, h, 16, 0.0, kind[b0:b1].contiguous(), coef[b0:b1].contiguous(),
                    eps[b0:b1].contiguous(), None, 2, L[b0:b1].contiguous(),
                    H[b0:b1].contiguous(), *src, ld, nt[b0:b1].contiguous(), pu, pl, keep, pn)
        ctx.check("compose")
        # in place, what lies past an item's terms is not the composition's
        live = torch.arange(keep, device="cuda")[None, :, None] < pn[:, None, :]
        return torch.where(live, pu, 0), torch.where(live, pl, 0), pn

    whole = run(0, B)
    step = 300                                         # few enough for the blocks alone
    parts = [run(b, min(B, b + step)) for b in range(0, B, step)]
    for a, p in zip(whole, zip(*parts)):
        assert torch.equal(a, torch.cat(p))
    assert bool(torch.isfinite(whole[0]).all())
    ctx.close()
