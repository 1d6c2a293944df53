"""The inversion of the aux Dyson equation (gw_aux_dyson) at the sizes where its route changes: in shared
memory below 80, panels of 16 columns with tensor-core updates up to 800, of 8 above; remainders of panels
and row tiles; matrices that need row interchanges; a singular one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _solve(gw, m):
    """(I - P0)^-1 - I for I - P0 = m [nw][n][n] through gw_aux_dyson."""
    nw, n = m.shape[:2]
    ctx = gw.gw_create((1, 1, 1), 2, n, nw, 10.0)
    assert ctx.nwb == nw
    P0 = torch.from_numpy(np.eye(n) - m).cuda()[None].contiguous()
    Pw = torch.empty_like(P0)
    gw.gw_aux_dyson(ctx, P0, Pw)
    try:
        gw.gw_synchronize(ctx)
        gw.gw_check_guards(ctx)
        return Pw.cpu().numpy()[0]
    finally:
        ctx.destroy()


@pytest.mark.parametrize("n", [1, 15, 32, 33, 79, 80, 81, 127, 200, 257, 480, 801])
def test_aux_dyson_inverts(n):
    """Random matrices (every column needs its pivot searched), one of them with a zero diagonal, and one
    with rows over six decades; backward error of the inverse as a partially pivoted elimination gives it."""
    from paper_2406_18479_gb300 import gw
    rng = np.random.default_rng(n)
    m = rng.standard_normal((3, n, n)) + 1j * rng.standard_normal((3, n, n))
    if n > 1:
        m[1] -= np.diag(np.diagonal(m[1]))
        m[2] *= 10.0 ** rng.uniform(-3, 3, (n, 1))
    x = _solve(gw, m) + np.eye(n)
    for a, b in zip(m, x):
        cond = np.linalg.norm(a, 2) * np.linalg.norm(np.linalg.inv(a), 2)
        # |A X - I| <= c n eps cond(A), c = 4 covers the growth of these matrices; the input I - P0 itself is rounded
        assert np.linalg.norm(a @ b - np.eye(n), 2) <= 4 * n * 2.0 ** -53 * cond * max(1.0, 2.0 / np.abs(a).max())


@pytest.mark.parametrize("n", [40, 96])
def test_singular_matrix_is_reported(n):
    from paper_2406_18479_gb300 import gw
    m = np.zeros((3, n, n), complex)
    m[:] = np.eye(n)
    m[1, :, n // 2] = 0.0
    with pytest.raises(gw.GWError):
        _solve(gw, m)
