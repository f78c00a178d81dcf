"""bern_linearize at orders below the variables: the fit block holds terms up to the
order only, and the bound it makes still lies outside the polynomial."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2211_14438_gb300 import bern

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,D,order", [(2, 2, 1), (3, 3, 1), (3, 3, 2), (4, 4, 2), (5, 5, 2),
                                       (2, 16, 1), (6, 3, 1)])
def test_fit_below_the_variables_is_sound(n, D, order):
    B, h = 2, 5
    M, Ml = bern.num_monomials(n, D), bern.num_monomials(n, min(n, order))
    rng = np.random.default_rng(100 * n + 10 * D + order)
    up = rng.normal(size=(B, M, h)).astype(np.float32)
    ex = bern.monomials(n, D).astype(int)
    up[0, :, 0] = (ex.max(1) <= 1) & (ex.sum(1) == min(n, D))     # the product of all variables
    lo = (up - rng.random((B, M, h)) * 0.01).astype(np.float32)
    nt = np.full((B, h), M, np.int32)
    t = [torch.from_numpy(x.copy()).cuda() for x in (up, lo, nt)]
    lu = torch.zeros(B, Ml, h, device="cuda")
    ll, r = torch.zeros_like(lu), torch.zeros(2, B, h, device="cuda")
    ln = torch.zeros(B, h, dtype=torch.int32, device="cuda")
    ctx = bern.Context(0)
    ctx.linearize(n, B, h, order, 0, t[0], t[1], M, t[2], lu, ll, Ml, ln, r[0], r[1])
    ctx.check("linearize")
    ctx.close()
    assert np.all(ln.cpu().numpy() == min(M, Ml))
    pts = np.vstack([rng.random((200, n)), np.zeros(n), np.ones(n), np.eye(n)])
    mono = np.prod(pts[:, None, :] ** ex[None], axis=2)
    for src, lin, sign in ((up, lu, 1), (lo, ll, -1)):
        lin = lin.cpu().numpy().astype(np.float64)
        for b, m in np.ndindex(B, h):
            want = mono @ src[b, :, m].astype(np.float64)
            got = mono[:, :Ml] @ lin[b, :, m]
            assert np.all(sign * (got - want) >= -1e-12 * np.abs(src[b, :, m]).sum()), (b, m, sign)
