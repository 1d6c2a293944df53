"""FP64 products on the tensor cores (csrc/k_oz64.cu) through the public calls that run on them: the
transforms against an extended-precision product, the FP64 contractions against the oracle, at the
edges of tiles, k-steps, exact chunks, split K and workspace pieces; non-finite and extreme values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _gw():
    from paper_2406_18479_gb300 import gw
    return gw


# a correctly summed product rounds once (2^-53 of the result) and carries 2^-59 of the row scales per
# term; an FP64 sum of K terms is allowed 2^-53 K. 8 x 2^-53 of sum |F||x| covers the first only.
TOL = 8 * 2.0 ** -53


@pytest.mark.parametrize("ntau", [9, 15, 16, 33, 64, 65, 100, 129, 200])
@pytest.mark.parametrize("nelem", [17, 64, 65, 1000])
def test_transform_matches_extended_precision(ntau, nelem):
    """to_matsubara and to_tau against long double, K below / at / above a k-step and the exact chunk."""
    gw = _gw()
    rng = np.random.default_rng(ntau * 1000 + nelem)
    ctx = gw.gw_create((1, 1, 1), 4, 16, ntau, 20.0)
    _, _, F, B = gw.gw_grid_build(ntau, 20.0, 0)
    for M, call in ((F, gw.gw_to_matsubara), (B, gw.gw_to_tau)):
        x = rng.standard_normal((2, M.shape[1], nelem)) + 1j * rng.standard_normal((2, M.shape[1], nelem))
        x *= np.exp(-rng.uniform(0, 12, (2, M.shape[1], 1)))
        X = torch.from_numpy(x).cuda()
        Y = torch.empty((2, M.shape[0], nelem), dtype=torch.complex128, device="cuda")
        call(ctx, 0, X, Y)
        gw.gw_synchronize(ctx)
        y = Y.cpu().numpy()
        L = np.longdouble
        for b in range(2):
            re = M.real.astype(L) @ x[b].real.astype(L) - M.imag.astype(L) @ x[b].imag.astype(L)
            im = M.real.astype(L) @ x[b].imag.astype(L) + M.imag.astype(L) @ x[b].real.astype(L)
            bound = TOL * (np.abs(M) @ np.abs(x[b])) + 2.0 ** -50 * M.shape[1] * 2.0 ** -8 * \
                np.abs(M).max(1)[:, None] * np.abs(x[b]).max(0)[None, :]
            assert np.all(np.abs(y[b].real - re) <= bound) and np.all(np.abs(y[b].imag - im) <= bound)
    gw.gw_check_guards(ctx)
    ctx.destroy()


def test_transform_special_values():
    """Infinities, NaN, zeros and magnitudes beyond the digit range behave as an FP64 sum does."""
    gw = _gw()
    T, n = 40, 80
    rng = np.random.default_rng(5)
    _, _, F, _ = gw.gw_grid_build(T, 20.0, 0)
    x = rng.standard_normal((1, T, n)) + 1j * rng.standard_normal((1, T, n))
    x[0, 3, 0] = np.inf
    x[0, 4, 1] = np.nan
    x[0, :, 2] = 0.0
    x[0, :, 3] *= 1e-200
    x[0, :, 4] *= 1e200
    x[0, :, 5] *= 1e-306
    ctx = gw.gw_create((1, 1, 1), 4, 16, T, 20.0)
    Y = torch.empty((1, ctx.nwb, n), dtype=torch.complex128, device="cuda")
    gw.gw_to_matsubara(ctx, 0, torch.from_numpy(x).cuda(), Y)
    gw.gw_synchronize(ctx)
    y = Y.cpu().numpy()[0]
    assert not np.isfinite(y[:, :2]).any() and np.isnan(y[:, 1]).all()
    assert np.all(y[:, 2] == 0)
    ref = F @ x[0][:, 3:]
    scale = np.abs(F) @ np.abs(x[0][:, 3:])
    assert np.all(np.abs(y[:, 3:] - ref) <= 2 * T * 2.0 ** -53 * scale + 1e-320)
    ctx.destroy()


@pytest.mark.parametrize("nk3,nao,naux,ntau,chunk", [
    ((1, 1, 1), 9, 36, 12, 0),        # one tile, split K
    ((1, 1, 1), 33, 130, 7, 0),       # row tiles with remainders
    ((2, 1, 1), 17, 65, 10, 3),       # uneven tau batches
    ((2, 2, 1), 12, 64, 9, 0),
    ((1, 1, 1), 70, 70, 5, 1),        # more orbitals than a row tile; digits made in pieces
])
def test_fp64_contractions_match_oracle(nk3, nao, naux, ntau, chunk):
    """P0 and Sigma of the FP64 precision against the oracle, to a few roundings of the largest element."""
    gw = _gw()
    from oracle import gw as O
    from paper_2406_18479_gb300 import inputs as I
    w = I.Workload("t", nk3, nao, naux, ntau, ntau, 10.0, 0.0, naux / 4.0, nao, solid=nk3 != (1, 1, 1))
    h, v, g = I.make_inputs(w)
    ref = O.sigma_eval(v, g, nk3, w.beta, spin_factor=2.0)
    ctx = gw.gw_create(nk3, nao, naux, ntau, w.beta, tau_chunk=chunk)
    V, Gt = torch.from_numpy(v).cuda(), torch.from_numpy(g).cuda()
    gw.gw_set_coulomb(ctx, V)
    P = torch.empty(ctx.shapes()["Pt"], dtype=torch.complex128, device="cuda")
    S = torch.empty(ctx.shapes()["Sig"], dtype=torch.complex128, device="cuda")
    gw.gw_polarization(ctx, Gt, P)
    p0 = P.cpu().numpy()
    assert np.abs(p0 - ref["P0t"]).max() <= 1e-13 * np.abs(ref["P0t"]).max()
    gw.gw_self_energy(ctx, Gt, torch.from_numpy(np.ascontiguousarray(ref["Pt"])).cuda(), S)
    gw.gw_synchronize(ctx)
    assert np.abs(S.cpu().numpy() - ref["Sig"]).max() <= 1e-13 * np.abs(ref["Sig"]).max()
    gw.gw_check_guards(ctx)
    ctx.destroy()


@pytest.mark.parametrize("nk3,nao,naux,ntau", [((2, 1, 1), 26, 104, 24), ((3, 1, 1), 27, 70, 30), ((1, 1, 1), 54, 60, 100),
                                               ((3, 1, 1), 40, 80, 40), ((1, 1, 1), 70, 100, 99)])
def test_static_exchange_matches_oracle(nk3, nao, naux, ntau):
    """Sigma^inf with its exchange on the tensor cores (from 2^26 multiply-adds on: the last two sizes, both
    sides of the fused kernel's nao limit, the last one in pieces of Q) or not, full and
    packed V, against the oracle; the two layouts agree bit for bit."""
    gw = _gw()
    from oracle import gw as O
    from paper_2406_18479_gb300 import inputs as I
    w = I.Workload("t", nk3, nao, naux, ntau, ntau, 10.0, 0.0, naux / 4.0, nao, solid=nk3 != (1, 1, 1))
    h, v, g = I.make_inputs(w)
    # the density is the library's: its extrapolation to beta has its own rounding (1e-12 at 100 nodes)
    out, ref = [], None
    for precision, packed in (("fp64", False), ("bf16x4", False), ("bf16x4", True)):
        ctx = gw.gw_create(nk3, nao, naux, ntau, w.beta, precision=precision, v_packed=packed)
        V = torch.from_numpy(I.pack_v(v) if packed else v).cuda()
        gw.gw_set_coulomb(ctx, V)
        S = torch.empty(ctx.shapes()["H"], dtype=torch.complex128, device="cuda")
        gamma = torch.empty_like(S)
        gw.gw_density(ctx, torch.from_numpy(g).cuda(), gamma)
        gw.gw_sigma_inf(ctx, torch.from_numpy(g).cuda(), S)
        gw.gw_synchronize(ctx)
        gw.gw_check_guards(ctx)
        if ref is None:
            ref = O.sigma_inf(v, gamma.cpu().numpy(), nk3, spin_factor=2.0)
        out.append(S.cpu().numpy())
        ctx.destroy()
    assert np.abs(out[0] - ref).max() <= 1e-13 * np.abs(ref).max()
    assert np.array_equal(out[1], out[2]) and np.array_equal(out[0], out[1])
