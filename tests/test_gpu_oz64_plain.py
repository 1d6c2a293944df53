"""Rows without a digit form (infinities, NaN, magnitudes beyond 2^+-480) inside long FP64 contractions: K over
several exact chunks, split over CTAs, added to an earlier k-point's part, operands cut into pieces. Their outputs
are what an FP64 sum gives, and no other output is touched by them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [(1, 33, 66, 4, 1), (2, 17, 65, 5, 2), (2, 33, 40, 3, 0), (1, 70, 70, 2, 1)]   # nk, nao, naux, ntau, tau_chunk


def _inputs(nk, nao, naux, ntau, rng):
    c = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)      # noqa: E731
    v = c(nk, nk, naux, nao, nao)
    return v + v.conj().transpose(1, 0, 2, 4, 3), c(nk, ntau, nao, nao), c(nk, ntau, naux, naux)


def _p0(v, g, q, t):
    """-(s / nk) sum_k A B^T of one (q, t), and the sum of the moduli of its terms."""
    nk, ntau, naux = len(g), g.shape[1], v.shape[2]
    val, mag = 0, 0
    for k in range(nk):
        p = (k + q) % nk
        a = (v[k, p] @ g[p, t]).reshape(naux, -1)
        b = (v[p, k] @ g[k, ntau - 1 - t]).transpose(0, 2, 1).reshape(naux, -1)
        ma = (np.abs(v[k, p]) @ np.abs(g[p, t])).reshape(naux, -1)
        mb = (np.abs(v[p, k]) @ np.abs(g[k, ntau - 1 - t])).transpose(0, 2, 1).reshape(naux, -1)
        val, mag = val - 2.0 / nk * (a @ b.T), mag + 2.0 / nk * (ma @ mb.T)
    return val, mag


def _sigma(v, g, p, k, t):
    nk, nao, naux = len(g), g.shape[2], v.shape[2]
    val, mag = 0, 0
    for q in range(nk):
        m = (k - q) % nk
        z = (v[k, m] @ g[m, t]).transpose(1, 0, 2).reshape(nao, -1)
        r = (p[q, t] @ v[m, k].reshape(naux, -1)).reshape(naux * nao, nao)
        mz = (np.abs(v[k, m]) @ np.abs(g[m, t])).transpose(1, 0, 2).reshape(nao, -1)
        mr = (np.abs(p[q, t]) @ np.abs(v[m, k]).reshape(naux, -1)).reshape(naux * nao, nao)
        val, mag = val - z @ r / nk, mag + mz @ mr / nk
    return val, mag


def _run(case, v, g, p):
    from paper_2406_18479_gb300 import gw
    nk, nao, naux, ntau, chunk = case
    ctx = gw.gw_create((nk, 1, 1), nao, naux, ntau, 10.0, tau_chunk=chunk)
    V, G = torch.from_numpy(v).cuda(), torch.from_numpy(g).cuda()
    gw.gw_set_coulomb(ctx, V)
    P = torch.empty(ctx.shapes()["Pt"], dtype=torch.complex128, device="cuda")
    S = torch.empty(ctx.shapes()["Sig"], dtype=torch.complex128, device="cuda")
    gw.gw_polarization(ctx, G, P)
    gw.gw_self_energy(ctx, G, torch.from_numpy(p).cuda(), S)
    gw.gw_synchronize(ctx)
    gw.gw_check_guards(ctx)
    ctx.destroy()
    return P.cpu().numpy(), S.cpu().numpy()


@pytest.mark.parametrize("case", CASES)
def test_extreme_rows(case):
    """Auxiliary functions scaled by 1e-200, 1e-160 and 1e148 in P0, tau nodes of P~ by 1e-180 and 1e160 in Sigma: each
    output within the rounding of its own terms (both sides: K terms, and the two products before them)."""
    nk, nao, naux, ntau, _ = case
    rng = np.random.default_rng(naux)
    v, g, p = _inputs(nk, nao, naux, ntau, rng)
    w = v.copy()
    w[:, :, 3] *= 1e-200
    w[:, :, naux // 2] *= 1e148
    w[:, :, naux - 1] *= 1e-160
    pt, _ = _run(case, w, g, p)
    for q in range(nk):
        val, mag = _p0(w, g, q, 0)
        bound = 2 * (2 * nao + nk * nao * nao + 4) * 2.0 ** -52 * mag + 1e-305
        assert np.all(np.abs(pt[q, 0] - val) <= bound)
    pp = p.copy()
    pp[:, 0] *= 1e-180
    pp[:, ntau - 1] *= 1e160
    _, s = _run(case, v, g, pp)
    for k in range(nk):
        for t in (0, ntau - 1):
            val, mag = _sigma(v, g, pp, k, t)
            assert np.all(np.abs(s[k, t] - val) <= 2 * (naux + nao + nk * naux * nao + 4) * 2.0 ** -52 * mag)


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_rows(case, bad):
    """One element of V: its auxiliary row and column of P0 are non-finite, everything else as without it. One
    element of P~: Sigma of its tau node is, the other nodes are bit for bit as without it."""
    nk, nao, naux, ntau, _ = case
    rng = np.random.default_rng(naux + 1)
    v, g, p = _inputs(nk, nao, naux, ntau, rng)
    clean, clean_s = _run(case, v, g, p)
    w = v.copy()
    w[0, 0, 5, 1, 2] = bad
    pt, _ = _run(case, w, g, p)
    hit = np.zeros((naux, naux), bool)
    hit[5] = hit[:, 5] = True
    assert not np.isfinite(pt[0, 0][hit]).any()
    assert np.array_equal(pt[0, 0][~hit], clean[0, 0][~hit])
    pp = p.copy()
    pp[0, 1, 2, 3] = bad
    _, s = _run(case, v, g, pp)
    assert not np.isfinite(s[:, 1]).any()
    keep = [t for t in range(ntau) if t != 1]
    assert np.array_equal(s[:, keep], clean_s[:, keep])


def test_more_left_outputs_than_a_list_holds():
    """Some rows of V beyond the digit range in every tile, over a hundred tiles a CTA: outputs in the list, those
    that find no room in it, against plain complex128 products on the device."""
    from paper_2406_18479_gb300 import gw
    nk, nao, naux, ntau = 8, 26, 104, 80
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    c = lambda *s: torch.view_as_complex(torch.randn(s + (2,), dtype=torch.float64, device="cuda", generator=gen))   # noqa: E731
    V, G = c(nk, nk, naux, nao, nao), c(nk, ntau, nao, nao)
    V[:, :, :, 0, :] *= 1e148
    ctx = gw.gw_create((2, 2, 2), nao, naux, ntau, 10.0)
    gw.gw_set_coulomb(ctx, V)
    P = torch.full(ctx.shapes()["Pt"], float("nan"), dtype=torch.complex128, device="cuda")
    gw.gw_polarization(ctx, G, P)
    gw.gw_synchronize(ctx)
    gw.gw_check_guards(ctx)
    ctx.destroy()
    for q, t in ((0, 3), (5, 0), (7, 39)):
        ref, mag = 0, 0
        for k in range(nk):
            p = k ^ q                                            # k + q on a mesh of twos
            f = lambda x, y: (x @ y).reshape(naux, -1)           # noqa: E731
            g = lambda x, y: (x @ y).transpose(1, 2).reshape(naux, -1)   # noqa: E731
            ref = ref - 2.0 / nk * f(V[k, p], G[p, t]) @ g(V[p, k], G[k, ntau - 1 - t]).T
            m = lambda x: torch.complex(x.abs(), torch.zeros_like(x.real))    # noqa: E731
            mag = mag + 2.0 / nk * (f(m(V[k, p]), m(G[p, t])) @ g(m(V[p, k]), m(G[k, ntau - 1 - t])).T).real
        bound = 2 * (2 * nao + nk * nao * nao + 4) * 2.0 ** -52 * mag
        assert bool(((P[q, t] - ref).abs() <= bound).all())
