"""The enclosure kernels without a grid (two and three variables up to order 8,
four and more up to order 10, order 1 everywhere) against the Bernstein
coefficients in float64, at the edges of their ranges: every variable count,
the smallest and largest orders, ragged term counts, orders below the degree,
item counts that are no multiple of a block's, and coefficients that are not
finite."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _graded(n, D):
    def of(n, d):
        if n == 1:
            return [(d,)]
        return [(a,) + t for a in range(d, -1, -1) for t in of(n - 1, d - a)]
    return np.array([e for d in range(D + 1) for e in of(n, d)])


def _range(n, l, e, a):
    """Bernstein coefficients of order l (Def. 2) of sum a t^e, e of degree <= l,
    with the other terms at their own intervals: (min, max)."""
    low = e.sum(1) <= l
    g = np.zeros((l + 1,) * n)
    for t, c in zip(e[low], a[low]):
        g[tuple(t)] = c / math.prod(math.comb(l, int(j)) for j in t)
    T = np.array([[math.comb(i, j) for j in range(l + 1)] for i in range(l + 1)], float)
    for _ in range(n):
        g = np.tensordot(g, T, axes=([0], [1]))
    r = a[~low]
    return g.min() + np.minimum(r, 0).sum(), g.max() + np.maximum(r, 0).sum()


@pytest.mark.parametrize("n,l,D,B,h", [
    (2, 2, 2, 3, 7), (2, 8, 8, 5, 33), (2, 5, 7, 2, 9), (3, 2, 2, 3, 43), (3, 4, 4, 2, 26),
    (3, 8, 8, 3, 15), (3, 7, 7, 1, 1), (3, 5, 6, 2, 11), (4, 2, 2, 2, 9), (4, 3, 3, 2, 5),
    (4, 4, 4, 2, 5), (4, 10, 10, 1, 2), (5, 2, 2, 2, 5), (5, 5, 5, 1, 3), (5, 6, 7, 1, 3),
    (6, 2, 2, 1, 7), (6, 4, 4, 1, 5), (6, 3, 4, 1, 3), (7, 2, 2, 1, 3), (7, 4, 4, 1, 2),
    (8, 2, 2, 1, 3), (8, 3, 3, 1, 2), (8, 1, 1, 2, 5), (5, 1, 2, 2, 5), (1, 1, 1, 2, 5)])
def test_enclose_orders(n, l, D, B, h):
    import torch
    from paper_2211_14438_gb300 import bern
    rng = np.random.default_rng(100 * n + 10 * l + D)
    e = _graded(n, D)
    M = len(e)
    up = rng.normal(size=(B, M, h)).astype(np.float32)
    lo = rng.normal(size=(B, M, h)).astype(np.float32)
    # near-linear neighbours of a vertex exercise the pruning, zero polynomials
    # and ragged counts the tables
    up[:, n + 1:, ::2] *= 0.01
    lo[:, n + 1:, ::2] *= 0.01
    nt = rng.integers(1, M + 1, (B, h)).astype(np.int32)
    nt[:, ::3] = M
    nt.reshape(-1)[-1] = 0
    ctx = bern.Context(0)
    dev = [torch.from_numpy(x).cuda() for x in (up, lo, nt)]
    rl, ru = torch.zeros(B, h, device="cuda"), torch.zeros(B, h, device="cuda")
    ctx.enclose(n, B, h, l, 0, dev[0], dev[1], M, dev[2], rl, ru)
    ctx.check("enclose")
    rl, ru = rl.cpu().numpy().astype(np.float64), ru.cpu().numpy().astype(np.float64)
    for b in range(B):
        for m in range(h):
            k = nt[b, m]
            au, al = up[b, :k, m].astype(np.float64), lo[b, :k, m].astype(np.float64)
            hi, lw = _range(n, l, e[:k], au)[1], _range(n, l, e[:k], al)[0]
            # every coefficient is a sum with weights in [0, 1]; a pass adds at
            # most l roundings of 2^-23, the scaling two, the other terms M
            tol = (n * l + M + 4) * 2.0 ** -23
            assert hi - 1e-12 <= ru[b, m] <= hi + tol * (np.abs(au).sum() + 1e-30), (b, m)
            assert lw + 1e-12 >= rl[b, m] >= lw - tol * (np.abs(al).sum() + 1e-30), (b, m)
    ctx.close()


@pytest.mark.parametrize("n,l", [(2, 4), (3, 4), (4, 3), (5, 2), (6, 4), (6, 1)])
def test_enclose_non_finite_coefficients_are_reported(n, l):
    import torch
    from paper_2211_14438_gb300 import bern
    M = len(_graded(n, l))
    for bad in (float("inf"), float("nan")):
        up = torch.ones(1, M, 4, device="cuda")
        lo = -torch.ones(1, M, 4, device="cuda")
        up[0, 0, 1] = bad
        lo[0, 0, 2] = -bad
        nt = torch.full((1, 4), M, dtype=torch.int32, device="cuda")
        rl, ru = torch.zeros(1, 4, device="cuda"), torch.zeros(1, 4, device="cuda")
        ctx = bern.Context(0)
        ctx.enclose(n, 1, 4, l, 0, up, lo, M, nt, rl, ru)
        assert ctx.sync() == bern.BERN_E_NONFINITE
        # the other items keep their values
        assert np.isfinite(ru.cpu().numpy()[0, [0, 2, 3]]).all()
        assert np.isfinite(rl.cpu().numpy()[0, [0, 1, 3]]).all()
        ctx.close()
