"""The Horner kernel of several items a warp on coefficients that round: every
coefficient but the constant equals that of the block form bit for bit (the same
products in the same order, packed with swapped ends or not), the constants differ
by the order of their sums only, and both bounds lie on the sound side of the
composition in float64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2211_14438_gb300 import bern

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,D,d,cap", [
    (2, 1, 3, 16), (2, 2, 3, 16), (2, 4, 4, 16), (2, 4, 4, 9), (3, 2, 3, 16), (3, 2, 4, 5),
    (3, 5, 3, 16), (4, 2, 3, 16), (1, 3, 5, 16)])
def test_rounding(n, D, d, cap):
    B, h, part = 300, 41, 50                       # 12,300 neurons, 2050 in a slice
    M, keep = bern.num_monomials(n, D), bern.num_monomials(n, min(d * D, cap))
    rng = np.random.default_rng(1000 * n + 100 * D + 10 * d + cap)
    up = (rng.normal(size=(B, M, h)) * 0.5).astype(np.float32)
    lo = (up - rng.random((B, M, h)) * 0.1).astype(np.float32)
    nt = rng.choice([M, M, M - 1, max(1, n + 1)], (B, h)).astype(np.int32)
    live = np.arange(M)[None, :, None] < nt[:, None, :]
    mag = np.maximum(np.abs(np.where(live, up, 0)), np.abs(np.where(live, lo, 0)))[:, 1:].sum(1)
    L = (np.minimum(up[:, 0], lo[:, 0]) - mag - 0.1).astype(np.float32)
    H = (np.maximum(up[:, 0], lo[:, 0]) + mag + 0.1).astype(np.float32)
    a = rng.normal(size=(B, h, d + 1))
    coef = np.zeros((B, h, bern.COEF_STRIDE), np.float32)
    coef[..., :d + 1] = a
    eps = (rng.random((B, h)) * 0.01).astype(np.float32)
    dg = rng.integers(max(3, d - 1), d + 1, (B, h)).astype(np.uint8)   # order 2: a2 >= 0 only
    ctx = bern.Context(0)
    kinds = [np.full((B, h), 2, np.int8), np.where(rng.random((B, h)) < 0.1, 2, 1).astype(np.int8)]
    for kind in kinds:
        def run(sl):
            t = [torch.from_numpy(np.ascontiguousarray(v[sl])).cuda()
                 for v in (kind, coef, eps, dg, L, H, up, lo, nt)]
            nb = len(t[8])
            pu = torch.zeros(nb, max(keep, M), h, device="cuda")
            pl = torch.zeros_like(pu)
            pn = torch.zeros(nb, h, dtype=torch.int32, device="cuda")
            ctx.compose(n, nb, h, cap, 0.0, t[0], t[1], t[2], t[3], d, t[4], t[5], t[6], t[7], M,
                        t[8], pu, pl, pu.shape[1], pn)
            ctx.check("compose")
            return [x.cpu().numpy() for x in (pu, pl, pn)]
        wu, wl, wn = run(slice(0, B))
        for s in range(0, B, part):
            su, sl_, sn = run(slice(s, s + part))
            assert np.array_equal(sn, wn[s:s + part])
            for x, y in ((su, wu[s:s + part]), (sl_, wl[s:s + part])):
                assert np.array_equal(x[:, 1:], y[:, 1:])
                # the constant holds sums of up to `full` dropped terms and the shift by
                # 5 u ||s||_1 (M terms), each rounded once per term in either order
                full = bern.num_monomials(n, d * D)
                size = 1 + np.abs(y).sum(1) + (np.abs(coef).sum(2) * (1 + mag) ** d)[s:s + part]
                assert np.all(np.abs(x[:, 0] - y[:, 0]) <=
                              2.0 ** -22 * (full - min(full, keep) + M + 4) * size)
        # sound at random points, the vertices 0 and 1 among them
        ex = bern.monomials(n, min(d * D, cap)).astype(int)
        pts = rng.random((24, n))
        pts[0], pts[1] = 0.0, 1.0
        mono = np.prod(pts[:, None, :] ** ex[None], axis=2)
        for b, m in zip(rng.integers(0, B, 60), rng.integers(0, h, 60)):
            if kind[b, m] != 2:
                continue
            k, dd = nt[b, m], int(dg[b, m])
            c = coef[b, m, :dd + 1].astype(np.float64)
            kk = wn[b, m]
            for src, out, upper in ((up, wu, True), (lo, wl, False)):
                p = mono[:, :k] @ src[b, :k, m].astype(np.float64)
                s = (p - float(L[b, m])) / (float(H[b, m]) - float(L[b, m]))
                want = np.polynomial.polynomial.polyval(s, c) - (0 if upper else float(eps[b, m]))
                got = mono[:, :kk] @ out[b, :kk, m].astype(np.float64)
                tiny = 1e-12 * (1 + np.abs(out[b, :kk, m]).sum())
                assert np.all(got >= want - tiny if upper else got <= want + tiny), (b, m, upper)
    ctx.close()
