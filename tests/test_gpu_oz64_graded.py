"""FP64 products on the tensor cores whose operands are graded: where the large elements of one meet the
small ones of the other, the digits of a row hold too little and the result still has the error bound of an
FP64 sum, K 2^-52 sum |a| |b| (complex K; the factor 2 of a complex multiply-add included)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
LC = np.clongdouble


def _gw():
    from paper_2406_18479_gb300 import gw
    return gw


def _mod(x):
    return np.abs(x).astype(np.longdouble)


@pytest.mark.parametrize("ntau", [15, 16, 33, 64, 65, 129])
@pytest.mark.parametrize("nelem", [33, 65])
@pytest.mark.parametrize("own", [False, True])
def test_transform_of_graded_input(ntau, nelem, own):
    """Elements that grow or fall over the nodes by up to 2^30, sit on one node, or cancel the matrix row
    by row, both directions; compared output by output."""
    gw = _gw()
    rng = np.random.default_rng(ntau + nelem)
    ctx = gw.gw_create((1, 1, 1), 4, 16, ntau, 20.0)
    tau = gw.gw_grid_build(ntau, 20.0, 0)[0]
    grids = [gw.gw_grid_build(ntau, 20.0, stat)[2:] for stat in (0, 1)]
    if own:      # a caller's grid: nodes towards the ends count up to 2^50 less, inputs there up to 2^60 more
        c = 2.0 ** (-50.0 * np.abs(np.linspace(-1, 1, ntau)))
        grids = [(F * c, B / c[:, None]) for F, B in grids]
        om = [(2 * gw.gw_grid_build(ntau, 20.0, s)[1] + s) * np.pi / 20.0 for s in (0, 1)]
        gw.gw_set_grids(ctx, tau, *grids[0], *grids[1], om[1], om[0])
    for stat in (0, 1):
        F, B = grids[stat]
        for M, call in ((F, gw.gw_to_matsubara), (B, gw.gw_to_tau)):
            n = M.shape[1]
            x = rng.standard_normal((2, n, nelem)) + 1j * rng.standard_normal((2, n, nelem))
            slope = rng.uniform(-30, 30, (2, 1, nelem))
            x *= 2.0 ** (slope * np.linspace(0, 1, n)[None, :, None])
            x[1, :, ::3] *= (2.0 ** -40) ** (np.arange(n)[:, None] != rng.integers(0, n, x[1, :, ::3].shape[1]))
            if own and M is F:
                x /= c[None, :, None] ** 1.2
            small = np.abs(M).min(0) < 1e-2 * np.abs(M).max(0)     # nodes with a small entry in some row
            if small.any():
                x[1, ~small, 1::3] *= 2.0 ** -40
            X = torch.from_numpy(x).cuda()
            Y = torch.empty((2, M.shape[0], nelem), dtype=torch.complex128, device="cuda")
            call(ctx, stat, X, Y)
            gw.gw_synchronize(ctx)
            y = Y.cpu().numpy()
            for b in range(2):
                ref = M.astype(LC) @ x[b].astype(LC)
                bound = n * 2.0 ** -52 * (_mod(M) @ _mod(x[b]))
                assert np.all(_mod(y[b] - ref) <= bound)
    gw.gw_check_guards(ctx)
    ctx.destroy()


def _graded(nk, nao, naux, ntau, rng):
    """V_ij rises as h_i h_j and G_ab falls as 1 / h_b^2, h from 1 to 2^30 over the basis: in P0 the sum over (d, b)
    is of terms 1 / (h_d h_b), its first operand as large as h_d / h_b^2 and its second as h_b / h_d^2."""
    h = 2.0 ** (30.0 * np.linspace(0, 1, nao))
    v = rng.standard_normal((nk, nk, naux, nao, nao)) + 1j * rng.standard_normal((nk, nk, naux, nao, nao))
    v = (v + v.conj().transpose(1, 0, 2, 4, 3)) * h[:, None] * h
    g = (rng.standard_normal((nk, ntau, nao, nao)) + 1j * rng.standard_normal((nk, ntau, nao, nao))) / h ** 2
    return v, g


@pytest.mark.parametrize("nk,nao,naux,ntau,chunk", [(1, 12, 40, 6, 0), (1, 33, 66, 4, 1), (2, 17, 65, 5, 2), (1, 70, 70, 2, 1)])
def test_contractions_of_graded_operands(nk, nao, naux, ntau, chunk):
    """P0 and Sigma, FP64: sum over (d, b) or (Q, b) with the grading in opposite directions, K below and above
    an exact chunk, split over CTAs and cut into pieces."""
    gw = _gw()
    rng = np.random.default_rng(nao)
    v, g = _graded(nk, nao, naux, ntau, rng)
    p = rng.standard_normal((nk, ntau, naux, naux)) + 1j * rng.standard_normal((nk, ntau, naux, naux))
    p *= 2.0 ** (-30.0 * np.linspace(0, 1, naux))[None, None, :, None]
    ctx = gw.gw_create((nk, 1, 1), nao, naux, ntau, 10.0, tau_chunk=chunk)
    V, G = torch.from_numpy(v).cuda(), torch.from_numpy(g).cuda()
    gw.gw_set_coulomb(ctx, V)
    P = torch.empty(ctx.shapes()["Pt"], dtype=torch.complex128, device="cuda")
    S = torch.empty(ctx.shapes()["Sig"], dtype=torch.complex128, device="cuda")
    gw.gw_polarization(ctx, G, P)
    gw.gw_self_energy(ctx, G, torch.from_numpy(p).cuda(), S)
    gw.gw_synchronize(ctx)
    gw.gw_check_guards(ctx)
    got_p, got_s = P.cpu().numpy(), S.cpu().numpy()
    ctx.destroy()

    def gemm(a, b):       # value in extended precision, and sum |a| |b|
        return a[0] @ b[0], a[1] @ b[1]

    def pair(x):
        return x.astype(LC), _mod(x)

    rows, cols = rng.permutation(naux)[:8], rng.permutation(naux)[:24]                   # Q, Q' and j compared
    js = rng.permutation(nao)[:8]
    for t in ((0,) if nk > 1 else (0, ntau // 2)):
        q = 0
        ref, mag = 0, 0
        for k in range(nk):
            A = gemm(pair(v[k, k][rows]), pair(g[k, t]))                                 # [Q][d][b]
            D = gemm(pair(v[k, k][cols]), pair(g[k, ntau - 1 - t]))                      # [Q'][b][d]
            a = [z.reshape(len(rows), -1) for z in A]
            d = [z.transpose(0, 2, 1).reshape(len(cols), -1) for z in D]
            r, m = gemm(a, [z.T for z in d])
            ref, mag = ref - 2.0 / nk * r, mag + 2.0 / nk * m
        # the roundings of both V.G products and of the sum itself
        bound = (2 * nao + nk * nao * nao + 4) * 2.0 ** -52 * mag
        assert np.all(_mod(got_p[q, t][np.ix_(rows, cols)] - ref) <= bound)
    for t in (0, ntau - 1):
        k = 0
        ref, mag = 0, 0
        for q in range(nk):
            m_ = (k - q) % nk
            R = gemm(pair(p[q, t]), pair(v[m_, k][:, :, js].reshape(naux, -1)))          # [Q][(b j)]
            Z = gemm(pair(v[k, m_]), pair(g[m_, t]))                                     # [Q][i][b]
            r, m = gemm([z.transpose(1, 0, 2).reshape(nao, -1) for z in Z], [z.reshape(naux * nao, len(js)) for z in R])
            ref, mag = ref - r / nk, mag + m / nk
        bound = (naux + nao + nk * naux * nao + 4) * 2.0 ** -52 * mag
        assert np.all(_mod(got_s[k, t][:, js] - ref) <= bound)


def _eliminate(a):
    """Inverse by Gauss-Jordan with partial pivoting, column by column, in the type of a."""
    a, n, swaps = a.copy(), len(a), []
    for j in range(n):
        p = j + int(np.argmax(np.abs(a[j:, j])))
        swaps.append(p)
        a[[j, p]] = a[[p, j]]
        inv = 1 / a[j, j]
        row = a[j] * inv
        row[j] = inv
        f = a[:, j].copy()
        f[j] = 0
        a[:, j] = 0
        a -= np.outer(f, row)
        a[j] = row
    for c in range(n - 1, -1, -1):
        a[:, [c, swaps[c]]] = a[:, [swaps[c], c]]
    return a


@pytest.mark.parametrize("n", [80, 96, 161])
def test_inverse_of_weakly_coupled_blocks(n):
    """Two systems with a coupling of 1e-10, the border inside a panel: the coupling entries of the inverse are as
    accurate, each relative to itself, as those of a column-by-column elimination (the median of them: a few are
    small by cancellation; eight times covers the order of the sums)."""
    gw = _gw()
    rng = np.random.default_rng(n)
    m = rng.standard_normal((3, n, n)) + 1j * rng.standard_normal((3, n, n))
    h = n // 2 - 4
    m[:, :h, h:] *= 1e-10
    m[:, h:, :h] *= 1e-10
    m = np.eye(n) - (np.eye(n) - m)          # what the call inverts is I - P0, rounded
    ctx = gw.gw_create((1, 1, 1), 2, n, 3, 10.0)
    P0 = torch.from_numpy(np.eye(n) - m).cuda()[None].contiguous()
    Pw = torch.empty_like(P0)
    gw.gw_aux_dyson(ctx, P0, Pw)
    gw.gw_synchronize(ctx)
    gw.gw_check_guards(ctx)
    ctx.destroy()
    for a, y in zip(m, Pw.cpu().numpy()[0]):
        ref, plain = _eliminate(a.astype(LC)), _eliminate(a)
        for block in (np.s_[:h, h:], np.s_[h:, :h]):
            err = lambda z: float(np.median(_mod(z - ref)[block] / _mod(ref)[block]))      # noqa: E731
            assert err(y) <= 8 * err(plain) + 2.0 ** -44
