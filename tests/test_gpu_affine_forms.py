"""The forms of the affine step at the edges of their rules: the register-blocked
kernel's row tiles and live-input lists against the block tiles, a warp per box
against slices of the same call, and the quad kernel of narrow outputs against
float64.  The tiled forms add the same terms in the same order with the same
rounding, so they agree bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2211_14438_gb300 import bern
    c = bern.Context(0)
    yield c
    c.close()


def _problem(B, h_in, h_out, M, seed):
    rng = np.random.default_rng(seed)
    mid = rng.normal(size=(B, M, h_in)).astype(np.float32)
    gap = rng.random((B, M, h_in)).astype(np.float32)
    nt = rng.choice([0, 1, 2, M // 2, M - 1, M], size=(B, h_in)).astype(np.int32)
    nt = np.minimum(nt, M)
    nt[0, :] = np.minimum(nt[0, :], 1)                # a box without a live row
    nt[-1, :] = M                                     # and one of full inputs only
    past = np.arange(M)[None, :, None] >= nt[:, None, :]
    up = np.where(past, np.float32(1e30), mid + gap)  # never to be read
    lo = np.where(past, np.float32(-1e30), mid - gap)
    W = rng.normal(size=(h_out, h_in)).astype(np.float32)
    W[rng.random(W.shape) < 0.1] = 0.0
    b = rng.normal(size=h_out).astype(np.float32)
    return W, b, up, lo, nt


def _run(ctx, W, b, up, lo, nt):
    import torch
    B, M, h_in = up.shape
    h_out = len(W)
    d = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (W, b, up, lo, nt)]
    ou = torch.full((B, M, h_out), 7.0, device="cuda")
    ol = torch.full_like(ou, 7.0)
    on = torch.zeros(B, h_out, dtype=torch.int32, device="cuda")
    ctx.affine(B, h_out, h_in, d[0], d[1], d[2], d[3], M, d[4], ou, ol, M, on)
    assert ctx.sync() == 0
    return [x.cpu().numpy() for x in (ou, ol, on)]


@pytest.mark.parametrize("h_in,h_out,M,B", [
    (47, 64, 33, 3), (48, 32, 32, 3), (48, 33, 33, 3), (64, 64, 64, 3), (65, 100, 65, 3),
    (150, 70, 165, 2), (20, 40, 35, 3), (64, 64, 165, 1600)])
def test_wide_tiles_agree(ctx, h_in, h_out, M, B):
    p = _problem(B, h_in, h_out, M, h_in + M)
    got = {}
    try:
        for v in (1, 0, 2, 3):
            ctx.force_variant("affine", v)
            got[v] = _run(ctx, *p)
    finally:
        ctx.force_variant("affine", -1)
    for v in (0, 2, 3):
        for a, w in zip(got[v], got[1]):
            assert np.array_equal(a, w), v


@pytest.mark.parametrize("h_in,h_out,M", [(1, 17, 6), (20, 20, 15), (64, 31, 16)])
def test_a_warp_per_box_agrees_with_tiles(ctx, h_in, h_out, M):
    W, b, up, lo, nt = _problem(5000, h_in, h_out, M, h_in + M)
    whole = _run(ctx, W, b, up, lo, nt)
    for s in range(0, 5000, 500):
        part = _run(ctx, W, b, up[s:s + 500], lo[s:s + 500], nt[s:s + 500])
        for a, w in zip(part, whole):
            assert np.array_equal(a, w[s:s + 500])


@pytest.mark.parametrize("h_out", [1, 2, 3, 4])
@pytest.mark.parametrize("h_in,M,B", [(4, 1, 3), (8, 35, 3), (20, 33, 2), (64, 165, 3),
                                      (100, 7, 2), (128, 130, 2)])
def test_narrow_quads(ctx, h_in, M, B, h_out):
    W, b, up, lo, nt = _problem(B, h_in, h_out, M, h_in * h_out + M)
    ou, ol, on = _run(ctx, W, b, up, lo, nt)
    past = np.arange(M)[None, :, None] >= nt[:, None, :]
    u = np.where(past, 0.0, up).astype(np.float64)
    l = np.where(past, 0.0, lo).astype(np.float64)
    Wp, Wn = np.maximum(W, 0).astype(np.float64), np.minimum(W, 0).astype(np.float64)
    wu = u @ Wp.T + l @ Wn.T
    wl = l @ Wp.T + u @ Wn.T
    wu[:, 0] += b
    wl[:, 0] += b
    mag = np.maximum(np.abs(u), np.abs(l)) @ np.abs(W).T.astype(np.float64) + np.abs(b)
    # one directed rounding (2^-23) for each product and each partial sum, the
    # same again for a midpoint and a radius
    tol = 2.0 ** -23 * (2 * h_in + 8) * mag
    for k in range(B):
        Mb = max(1, int(nt[k].max()))
        assert np.all(on[k] == Mb)
        e = 1e-12 * mag[k, :Mb]
        assert np.all(ou[k, :Mb] >= wu[k, :Mb] - e) and np.all(ol[k, :Mb] <= wl[k, :Mb] + e)
        assert np.all(ou[k, :Mb] <= wu[k, :Mb] + tol[k, :Mb])
        assert np.all(ol[k, :Mb] >= wl[k, :Mb] - tol[k, :Mb])
