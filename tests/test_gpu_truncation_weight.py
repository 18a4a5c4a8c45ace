"""The tensor-core truncation where every kept column carries weight: products
whose bond is exactly what D* holds, or is cut by it at a visible weight."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = 8


def _state(b, seed, fall=0.0):
    """Random right-canonical sites of bond b (4 next to the ends) whose values at
    the middle bond fall from 1 to 1/2, times exp(-fall) a value."""
    r = np.random.default_rng(seed)
    dims = [1, 4] + [b] * (L - 3) + [4, 1]
    w = [r.standard_normal((dims[i], 2, 2, dims[i + 1])) for i in range(L)]

    def move_left(lo):
        for i in range(L - 1, lo, -1):
            q, t = np.linalg.qr(w[i].reshape(dims[i], -1).T)
            w[i] = q.T.reshape(w[i].shape)
            w[i - 1] = np.tensordot(w[i - 1], t.T, 1)

    move_left(L // 2 - 1)
    for i in range(L // 2):
        q, t = np.linalg.qr(w[i].reshape(-1, dims[i + 1]))
        w[i] = q.reshape(w[i].shape)
        if i < L // 2 - 1:
            w[i + 1] = np.tensordot(t, w[i + 1], 1)
    s = np.linspace(1.0, 0.5, b) * np.exp(-fall * np.arange(b))
    w[L // 2 - 1] = w[L // 2 - 1] * s
    move_left(0)
    w[0] /= np.linalg.norm(w[0])
    return w


def _dense(sites):
    v = sites[0][0]
    for w in sites[1:]:
        v = np.einsum("stb,buvc->sutvc", v, w, optimize=True).reshape(
            v.shape[0] * 2, v.shape[1] * 2, w.shape[3])
    return v[:, :, 0]


def _middle_values(P):
    h = 2 ** (L // 2)
    return np.linalg.svd(P.reshape(h, h, h, h).transpose(0, 2, 1, 3).reshape(h * h, h * h),
                         compute_uv=False)


def _doubled(b, dstar, prec, sweeps, fall=0.0, **kw):
    """The engine's doubling of a state, the exact product, the counters."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_00142_gb300.build import build
    build()
    from paper_1801_00142_gb300.engine import XTRG
    sites = _state(b, 31 * b + dstar, fall)
    rho = _dense(sites)
    P = rho.T @ rho
    eng = XTRG.xxz(L, 1.0, 0.7, tau0=2.0 ** -4, dstar=dstar, sweeps=sweeps, prec=prec, **kw)
    eng.set_state(sites, 0.0, 1.0, right_canonical=True)
    eng.double()
    out, lnc, _ = eng.get_state()
    o, c = eng.observables(), eng.counters()
    eng.close()
    C = _dense(out) * np.exp(lnc)
    # every site but the first is right-orthonormal on its live rows, to what a
    # split may leave, and zero on the others
    for w in out[1:]:
        m = w.reshape(w.shape[0], -1)
        G = m @ m.T
        live = np.diag(G) > 0.5
        assert np.abs(G[np.ix_(live, live)] - np.eye(live.sum())).max() <= 1e-4
        assert not m[~live].any()
    assert c["exact_split_fallbacks"] <= 0.1 * c["two_site_updates"]
    return P, C, o, out


# bond of the state, D*, width of an orthonormalisation block: the product's bond
# b^2 fills D*, or leaves columns without weight up to the edge of a tile or panel
@pytest.mark.parametrize("b,dstar,block", [
    (8, 64, 0), (8, 64, 32), (8, 65, 0), (9, 81, 0), (10, 100, 0), (10, 100, 32), (11, 121, 0),
    (11, 127, 0), (11, 129, 0), (12, 144, 0), (13, 173, 0), (13, 173, 96), (14, 200, 0)])
@pytest.mark.parametrize("keep_parts", [True, False])
def test_no_column_of_weight_is_lost(b, dstar, block, keep_parts):
    """Nothing is cut, so the doubling equals the product.  Bound: a factor may be
    1e-4 from orthonormal before a split refuses it, which changes what it keeps
    by as much; each of the L - 1 splits adds noise of 1e-5 of the norm, 2.6e-5 in
    quadrature; the 4 L contractions are right to 2^-22 each (24-bit operands,
    FP32 sums), 8e-6.  1.5e-4 of the norm bounds them; one missing column of the
    middle bond is three to sixty times that."""
    P, C, o, out = _doubled(b, dstar, "bf16x6", 2, keep_parts=keep_parts, orth_block=block)
    n, s = np.linalg.norm(P), _middle_values(P)
    assert s[b * b - 1] > 5e-4 * n and (b * b >= 256 or s[b * b] < 1e-12 * n)
    assert np.linalg.norm(C - P) <= 1.5e-4 * n
    assert o["max_bond"] == dstar


@pytest.mark.parametrize("b,dstar", [(8, 64), (8, 65), (9, 81), (11, 127), (13, 173)])
def test_three_products_lose_no_column_of_weight(b, dstar):
    """As above with operands of two planes, right to 2^-16: 4 L 2^-16 = 5e-4."""
    P, C, o, out = _doubled(b, dstar, "bf16x3", 2)
    assert np.linalg.norm(C - P) <= 5e-4 * np.linalg.norm(P)


@pytest.mark.parametrize("b,dstar,block", [(12, 97, 0), (13, 128, 0), (13, 129, 32), (14, 160, 0)])
def test_cut_keeps_the_heaviest_columns(b, dstar, block):
    """D* cuts the middle bond, and only that.  What is lost is at least the exact
    tail of the product's spectrum.  Eight subspace steps (four sweeps) leave of
    a direction outside the cut, r times as heavy as the last one inside, r^8
    of its amplitude: one of r < 0.75 no more than 1 % of its weight, and one closer
    costs at most 1 - 0.75^2 of the weight it displaces: 1.5 times the tail
    bounds both."""
    P, C, o, out = _doubled(b, dstar, "bf16x6", 4, fall=0.05, orth_block=block)
    n, s = np.linalg.norm(P), _middle_values(P)
    tail = (s[dstar:] ** 2).sum() / n ** 2
    assert tail > 1e-6
    lost = (np.linalg.norm(C - P) / n) ** 2
    assert tail * (1 - 1e-4) <= lost <= 1.5 * tail
    assert 0.5 * tail <= o["trunc_err"] <= 1.5 * tail
