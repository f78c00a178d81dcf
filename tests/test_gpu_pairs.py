"""Order-2 compositions outside the squaring kernels' tables or without their
scratch (the pair-list kernel: degrees past 8, and long inputs of a context that
may keep none of them in device memory), and long squares in several passes of
a small scratch."""
import numpy as np
import pytest

from test_gpu_square import U, _graded, _square_index

pytestmark = pytest.mark.gpu


def _problem(n, D, B, h, cap):
    from paper_2211_14438_gb300 import bern
    rng = np.random.default_rng(1000 * n + 10 * D + cap)
    e = _graded(n, D)
    fall = (0.6 ** e.sum(1))[None, :, None]
    p = dict(up=rng.normal(size=(B, len(e), h)) * fall, lo=rng.normal(size=(B, len(e), h)) * fall,
             L=-1.0 - rng.random((B, h)), H=1.0 + rng.random((B, h)), eps=rng.random((B, h)))
    p = {k: v.astype(np.float32) for k, v in p.items()}
    p["nt"] = np.full((B, h), len(e), np.int32)
    p["nt"][:, 1::3] = len(_graded(n, D - 1)) + 1     # a ragged prefix of the same degree
    p["coef"] = np.zeros((B, h, bern.COEF_STRIDE), np.float32)
    p["coef"][..., 0] = 0.125
    p["coef"][..., 1:3] = rng.random((B, h, 2))
    p["kind"] = np.full((B, h), 2, np.int8)
    return p


def _run(n, D, B, h, cap, p, scratch=None):
    import torch
    from paper_2211_14438_gb300 import bern
    keep = len(_graded(n, min(2 * D, cap)))
    d = {k: torch.from_numpy(v).cuda() for k, v in p.items()}
    pu, pl = torch.zeros(B, keep, h, device="cuda"), torch.zeros(B, keep, h, device="cuda")
    pn = torch.zeros(B, h, dtype=torch.int32, device="cuda")
    ctx = bern.Context(0)
    if scratch is not None:
        ctx.set_square_scratch_limit(scratch)
    k0 = ctx.kernel_launches()
    ctx.compose(n, B, h, cap, 0.0, d["kind"], d["coef"], d["eps"], None, 2, d["L"], d["H"],
                d["up"], d["lo"], p["up"].shape[1], d["nt"], pu, pl, keep, pn)
    ctx.check("compose")
    k = ctx.kernel_launches() - k0
    ctx.close()
    return pu.cpu().numpy(), pl.cpu().numpy(), pn.cpu().numpy(), k


@pytest.mark.parametrize("n,D,cap,B,h,scratch", [
    (2, 9, 64, 2, 9, None), (2, 16, 64, 1, 7, None), (2, 16, 24, 1, 7, None),
    (1, 12, 24, 2, 5, None), (3, 9, 15, 1, 4, None), (5, 8, 16, 1, 3, 0), (6, 7, 11, 1, 3, 0)])
def test_pair_lists(n, D, cap, B, h, scratch):
    p = _problem(n, D, B, h, cap)
    pu, pl, pn, _ = _run(n, D, B, h, cap, p, scratch)
    ix, full = _square_index(n, D)
    kept, M = len(_graded(n, min(2 * D, cap))), len(_graded(n, D))
    assert np.all(pn == kept)
    for b, m in np.ndindex(B, h):
        a0, a1, a2 = (float(p["coef"][b, m, j]) for j in range(3))
        for got, P, sign in ((pu, p["up"], 1), (pl, p["lo"], -1)):
            s = np.where(np.arange(M) < p["nt"][b, m], P[b, :, m].astype(np.float64), 0.0)
            s[0] -= float(p["L"][b, m])
            s /= float(p["H"][b, m]) - float(p["L"][b, m])
            sq = np.bincount(ix, (s[:, None] * s[None]).ravel(), full)
            mag = np.bincount(ix, np.abs(s[:, None] * s[None]).ravel(), full)
            cnt = np.bincount(ix, minlength=full)
            want, size = a2 * sq, a2 * mag
            want[:M] += a1 * s
            size[:M] += a1 * np.abs(s)
            # s carries three roundings, a product sum one per pair, the rest three
            tol = 2 * U * (cnt + 12) * size + 1e-30
            v = got[b, :kept, m].astype(np.float64)
            assert np.all(np.abs(v[1:] - want[1:kept]) <= tol[1:kept]), (b, m, sign)
            # the constant: the shift by the rounding of s, and the dropped terms
            drop = want[kept:]
            l1 = np.abs(s).sum()
            eta = 5 * U * l1
            slack = (a1 + 2 * a2 * (1 + eta)) * eta
            c = want[0] + a0 + sign * (slack + np.maximum(sign * drop, 0).sum())
            if sign < 0:
                c -= float(p["eps"][b, m])
            at = tol[0] + tol[kept:].sum() + 2 * U * ((full - kept + 12) * (
                size[0] + np.abs(drop).sum() + a0 + 1.0 + slack) + M * slack)
            assert abs(v[0] - c) <= at, (b, m, sign, v[0], c, at)


@pytest.mark.parametrize("n,D,cap", [(5, 8, 16), (5, 8, 13), (6, 7, 16)])
def test_long_squares_in_several_passes(n, D, cap):
    B, h = 3, 45                                      # five groups of 32, the last one short
    p = _problem(n, D, B, h, cap)
    whole = _run(n, D, B, h, cap, p)
    parts = _run(n, D, B, h, cap, p, 900 << 10)       # one or two groups at a time
    assert parts[3] > whole[3]
    for a, b in zip(parts[:3], whole[:3]):
        assert np.array_equal(a, b)


def test_concave_polynomials_of_long_inputs():
    """A caller's coefficients with a_2 < 0: past shared memory such items take the
    pair lists, their neighbours the squares by tiles, both as without a scratch."""
    n, D, B, h = 5, 8, 2, 40
    p = _problem(n, D, B, h, 16)
    convex = _run(n, D, B, h, 16, p)                  # raises where an item is refused
    p["coef"][:, ::4, 2] *= -1.0
    got, lists = _run(n, D, B, h, 16, p), _run(n, D, B, h, 16, p, 0)
    for a, b, c in zip(got[:2], lists[:2], convex[:2]):
        assert np.array_equal(a[..., ::4], b[..., ::4])
        keep = np.arange(h) % 4 != 0
        assert np.array_equal(a[..., keep], c[..., keep])
        assert not np.array_equal(a[..., ::4], c[..., ::4])
