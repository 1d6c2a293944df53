"""The inversions of both Dyson equations on matrices that only a stable elimination inverts well: rows or
columns of different size, near-parallel columns, an ill-conditioned overlap. Each is held to the error of a column-by-column Gauss-Jordan elimination with partial pivoting in the same precision,
both against the elimination in extended precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _eliminate(a, dtype):
    """Inverse by Gauss-Jordan with partial pivoting, column by column, in dtype."""
    a = a.astype(dtype)
    n, swaps = len(a), []
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


def _gauss(rng, n):
    return rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))


def _matrix(kind, n, rng):
    a = _gauss(rng, n)
    if kind.startswith("columns") or kind.startswith("both"):
        a = a * 10.0 ** rng.uniform(-5, 5, n)
    if kind.startswith("rows") or kind.startswith("both"):
        a = a * 10.0 ** rng.uniform(-5, 5, (n, 1))
    if kind == "few rows":                      # fewer large rows than a panel has columns
        a[:5] *= 1e10
    if kind == "parallel":                      # two pairs of near-parallel columns in every panel
        for k in range(0, n - 3, 8):
            a[:, k + 1] = a[:, k] + 1e-6 * a[:, k + 1]
            a[:, k + 3] = a[:, k + 2] + 1e-6 * a[:, k + 3]
    return a


def _dyson(gw, m):
    n = m.shape[-1]
    ctx = gw.gw_create((1, 1, 1), 2, n, len(m), 10.0)
    P0 = torch.from_numpy(np.eye(n) - m).cuda()[None].contiguous()
    Pw = torch.empty_like(P0)
    gw.gw_aux_dyson(ctx, P0, Pw)
    gw.gw_synchronize(ctx)
    gw.gw_check_guards(ctx)
    ctx.destroy()
    return Pw.cpu().numpy()[0] + np.eye(n)


KINDS = ["random", "columns", "rows", "both", "few rows", "parallel"]


@pytest.mark.parametrize("n", [79, 80, 96, 161, 200])
def test_aux_dyson_as_accurate_as_an_elimination(n):
    """Every kind in one call, so that matrices of a launch differ. The error of an entry is taken relative to
    the largest entries of its row and column (rows, then columns scaled to one), which scaling does not change.
    Eight times the reference elimination's covers the
    order of its sums; below 2^-44 (1000 roundings) it is not held against it."""
    from paper_2406_18479_gb300 import gw
    rng = np.random.default_rng(n)
    m = np.stack([_matrix(k, n, rng) for k in KINDS] + [np.eye(n, dtype=complex)])
    # I - P0 is formed by the call: what it inverts is I - (I - m), rounded
    m = np.eye(n) - (np.eye(n) - m)
    x = _dyson(gw, m)
    for kind, a, y in zip(KINDS, m, x):
        ref = _eliminate(a, np.clongdouble)
        plain = _eliminate(a, np.complex128)
        # the call returns (I - P0)^-1 - I, and the identity is added back here: one rounding of 1 + |x| each
        shift = np.eye(n) * 2.0 ** -51 * (1 + np.abs(np.diagonal(ref)).astype(float))
        r = np.abs(ref).max(1, keepdims=True)
        s = (np.abs(ref) / r).max(0, keepdims=True)
        err = lambda z: float((np.maximum(np.abs(z - ref) - shift, 0) / r / s).max())      # noqa: E731
        assert err(y) <= 8 * err(plain) + 2.0 ** -44, kind


@pytest.mark.parametrize("nao", [80, 104])
@pytest.mark.parametrize("delta", [1e-3, 1e-4])
def test_dyson_with_an_ill_conditioned_overlap(nao, delta):
    """gw_dyson_G with Sigma = 0 in a basis of near-parallel pairs (cond(S) about 4 / delta^2):
    G(i w) = ((i w + mu) S - H)^-1, back on the tau grid; against the elimination in extended precision."""
    from paper_2406_18479_gb300 import gw
    rng = np.random.default_rng(nao)
    ntau, beta, mu = 12, 10.0, 0.05
    x = np.linalg.qr(_gauss(rng, nao))[0]
    x[:, 1::2] = x[:, ::2] + delta * x[:, 1::2]
    x /= np.linalg.norm(x, axis=0)
    h = np.diag(rng.uniform(-1.0, 1.0, nao))
    S, H = x.conj().T @ x, x.conj().T @ h @ x
    ctx = gw.gw_create((1, 1, 1), nao, 4, ntau, beta, mu=mu)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)[None]).cuda()                 # noqa: E731
    gw.gw_set_overlap(ctx, dev(S))
    G = torch.empty(ctx.shapes()["Sig"], dtype=torch.complex128, device="cuda")
    gw.gw_dyson_G(ctx, dev(H), torch.zeros_like(G), G)
    gw.gw_synchronize(ctx)
    got = G.cpu().numpy()[0]
    ctx.destroy()
    _, idx, _, B = gw.gw_grid_build(ntau, beta, 1)
    w = (2 * idx + 1) * np.pi / beta
    mats = [(1j * v + mu) * S - H for v in w]
    ref = np.stack([_eliminate(a, np.clongdouble) for a in mats]).reshape(len(w), -1)
    plain = np.stack([_eliminate(a, np.complex128) for a in mats]).reshape(len(w), -1)
    t = lambda z: (B.astype(np.clongdouble) @ z).reshape(got.shape)                        # noqa: E731
    ref, plain = t(ref), t(plain)
    err = lambda z: float(np.abs(z - ref).max() / np.abs(ref).max())                       # noqa: E731
    assert err(got) <= 8 * err(plain) + 2.0 ** -44


@pytest.mark.parametrize("n", [79, 80, 200, 480, 801])
def test_scaled_rows_and_columns_leave_the_backward_error(n):
    """A = diag(r) X diag(s), r and s over ten decades: Z = diag(s) A^-1 diag(r) inverts X as if it had not been
    scaled. |X Z - I| <= 4 n eps cond(X) as for the unscaled matrices of the plain inversion test; every route by n."""
    from paper_2406_18479_gb300 import gw
    rng = np.random.default_rng(n)
    r, s = np.ones((3, n, 1)), np.ones((3, 1, n))
    r[0], s[1] = 10.0 ** rng.uniform(-10, 0, (n, 1)), 10.0 ** rng.uniform(-10, 0, n)
    r[2], s[2] = 10.0 ** rng.uniform(-5, 0, (n, 1)), 10.0 ** rng.uniform(-5, 0, n)
    m = np.stack([_gauss(rng, n) for _ in range(3)]) * r * s
    m = np.eye(n) - (np.eye(n) - m)
    y = _dyson(gw, m)
    for i in range(3):
        x, z = m[i] / r[i] / s[i], s[i].T * y[i] * r[i].T
        cond = np.linalg.norm(x, 2) * np.linalg.norm(np.linalg.inv(x), 2)
        assert np.linalg.norm(x @ z - np.eye(n), 2) <= 4 * n * 2.0 ** -53 * cond
