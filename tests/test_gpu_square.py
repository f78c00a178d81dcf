"""The squaring kernels (order-2 compositions of input degree <= 8) against the
products in float64: every variable count, tiles and rows, the smallest and
largest degrees, inputs in shared memory and in the scratch, truncation, ragged
term counts, more than one group of 32 and a warp per group."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def _graded(n, D):
    def of(n, d):
        if n == 1:
            return [(d,)]
        return [(a,) + t for a in range(d, -1, -1) for t in of(n - 1, d - a)]
    return np.array([e for d in range(D + 1) for e in of(n, d)], np.int64)


def _square_index(n, D):
    e, f = _graded(n, D), _graded(n, 2 * D)
    w = (2 * D + 1) ** np.arange(n, dtype=np.int64)
    key = f @ w
    order = np.argsort(key)
    k = e @ w
    return order[np.searchsorted(key[order], (k[:, None] + k[None]).ravel())], len(f)


@pytest.mark.parametrize("n,D,cap,B,h,check", [
    (1, 1, 16, 2, 5, 10), (1, 8, 16, 2, 40, 20), (2, 8, 16, 2, 9, 18), (3, 0, 16, 1, 3, 3),
    (3, 3, 16, 2, 33, 20), (3, 5, 16, 2, 20, 20), (3, 8, 16, 2, 17, 10), (3, 8, 11, 2, 9, 8),
    (4, 6, 16, 1, 9, 6), (4, 8, 16, 1, 5, 4), (5, 4, 16, 1, 9, 6), (5, 5, 7, 1, 5, 4),
    (5, 7, 16, 1, 40, 3), (5, 8, 13, 1, 5, 2), (6, 4, 16, 1, 9, 4), (6, 6, 16, 2, 33, 2),
    (6, 8, 16, 1, 3, 1), (7, 3, 16, 1, 5, 3), (7, 5, 9, 1, 3, 2), (8, 2, 16, 1, 5, 4),
    (8, 4, 16, 1, 3, 1), (2, 1, 16, 1300, 64, 12), (3, 2, 3, 1300, 64, 12)])
def test_square(n, D, cap, B, h, check):
    import torch
    from paper_2211_14438_gb300 import bern
    rng = np.random.default_rng(1000 * n + 10 * D + cap)
    e = _graded(n, D)
    M, Mf = len(e), len(_graded(n, 2 * D))
    keep = len(_graded(n, min(2 * D, cap)))
    fall = (0.6 ** e.sum(1))[None, :, None]
    up = (rng.normal(size=(B, M, h)) * fall).astype(np.float32)
    lo = (rng.normal(size=(B, M, h)) * fall).astype(np.float32)
    nt = np.full((B, h), M, np.int32)
    if D > 1:   # a ragged prefix of the same degree, and a lower degree
        nt[:, 1::3] = len(_graded(n, D - 1)) + 1
        nt[:, 2::5] = len(_graded(n, D // 2))
    L = -1.0 - rng.random((B, h)).astype(np.float32)
    H = 1.0 + rng.random((B, h)).astype(np.float32)
    coef = np.zeros((B, h, bern.COEF_STRIDE), np.float32)
    coef[..., 0] = 0.125
    coef[..., 1] = rng.random((B, h)).astype(np.float32)
    coef[..., 2] = rng.random((B, h)).astype(np.float32)
    eps = rng.random((B, h)).astype(np.float32)
    kind = np.full((B, h), 2, np.int8)
    dev = {k: torch.from_numpy(v).cuda() for k, v in
           dict(up=up, lo=lo, nt=nt, L=L, H=H, coef=coef, eps=eps, kind=kind).items()}
    pu, pl = torch.zeros(B, keep, h, device="cuda"), torch.zeros(B, keep, h, device="cuda")
    pn = torch.zeros(B, h, dtype=torch.int32, device="cuda")
    ctx = bern.Context(0)
    ctx.compose(n, B, h, cap, 0.0, dev["kind"], dev["coef"], dev["eps"], None, 2, dev["L"],
                dev["H"], dev["up"], dev["lo"], M, dev["nt"], pu, pl, keep, pn)
    ctx.check("compose")
    pu, pl, pn = pu.cpu().numpy(), pl.cpu().numpy(), pn.cpu().numpy()
    index = {}
    flat = rng.permutation(B * h)[:check]
    flat[0], flat[-1] = 0, B * h - 1
    for b, m in zip(flat // h, flat % h):
        d = next(k for k in range(D + 1) if len(_graded(n, k)) >= nt[b, m])
        if d not in index:
            index[d] = _square_index(n, d)
        ix, full = index[d]
        kept = min(full, len(_graded(n, min(2 * d, cap))))
        assert pn[b, m] == kept
        Md = len(_graded(n, d))
        a0, a1, a2 = (float(coef[b, m, j]) for j in range(3))
        for got, P, sign in ((pu, up, 1), (pl, lo, -1)):
            s = np.where(np.arange(Md) < nt[b, m], P[b, :Md, m].astype(np.float64), 0.0)
            s[0] -= float(L[b, m])
            s /= float(H[b, m]) - float(L[b, m])
            sq = np.bincount(ix, (s[:, None] * s[None]).ravel(), full)
            mag = np.bincount(ix, np.abs(s[:, None] * s[None]).ravel(), full)
            cnt = np.bincount(ix, minlength=full)
            want = a2 * sq
            want[:Md] += a1 * s
            size = a2 * mag
            size[:Md] += a1 * np.abs(s)
            # s carries three roundings, a product sum one per pair, the rest three
            tol = 2 * U * (cnt + 12) * size + 1e-30
            v = got[b, :kept, m].astype(np.float64)
            assert np.all(np.abs(v[1:] - want[1:kept]) <= tol[1:kept]), (b, m, sign)
            drop = want[kept:]
            l1 = np.abs(s).sum()
            eta = 5 * U * l1
            slack = (a1 + 2 * a2 * (1 + eta)) * eta
            c = want[0] + a0 + sign * (slack + np.maximum(sign * drop, 0).sum())
            if sign < 0:
                c -= float(eps[b, m])
            at = tol[0] + tol[kept:].sum() + 2 * U * ((full - kept + 12) * (
                size[0] + np.abs(drop).sum() + a0 + 1.0 + slack) + Md * slack)
            assert abs(v[0] - c) <= at, (b, m, sign, v[0], c, at)
    ctx.close()
