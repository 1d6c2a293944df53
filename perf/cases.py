"""What a user of the GW library has it compute: the cases that its speed is measured on.

Each case goes through the public Python entry points of ``paper_2406_18479_gb300.gw`` on one
problem size. ``prepare`` makes the device arrays and the context (or batch) a program keeps over
a self-consistency run, ``run`` is one pass, ``exact`` is the same result from plain torch in
complex128, on the definitions (Eqs. tilde_P0_tau, P0t_to_P0w, tilde_P_omega, sigma_gw, dyson,
sigma_inf and sigma2 of arXiv 2406.18479).

Kinds of case, by the call they time:
  sigma         gw_sigma_eval, one whole self-energy evaluation
  batch         gw_batch.sigma_eval, many molecules at once (one captured graph)
  polarization  gw_polarization      V.G.V products and P0(tau)
  self_energy   gw_self_energy       Sigma from G, P~ and V
  screened      gw_screened_interaction   tau -> i Omega, (I - P0)^-1 P0, i Omega -> tau
  dyson         gw_dyson_G           the Dyson update of G
  static        gw_sigma_inf         Hartree and exchange
  gf2           gw_gf2_self_energy   the second-order self-energy
"""
import functools
import math

import numpy as np
import torch

from paper_2406_18479_gb300 import gw

C128 = torch.complex128
DEV = "cuda"
SPIN = 2.0
BATCH_BUDGET = 24 << 30     # device bytes a batch may plan with


def _case(kind, mesh, nao, naux, ntau, beta, precision="fp64", **more):
    return dict(kind=kind, n1=mesh[0], n2=mesh[1], n3=mesh[2], nao=nao, naux=naux, ntau=ntau, beta=float(beta),
                precision=precision, **more)


def listed():
    return [
        # the smallest system, in the default precision: a scGW loop on a small molecule, bound by launches
        dict(_case("sigma", (1, 1, 1), 8, 32, 32, 50.0), name="sigma_molecule_nao8"),
        # one iteration of the Si-like 3x3x3 solid (two atoms, DZVP-sized basis) on the tensor-core path
        dict(_case("sigma", (3, 3, 3), 26, 200, 100, 100.0, "bf16x4"), name="sigma_solid333_nao26_mixed"),
        # the two contractions at the 4x4x4 solid's orbital and auxiliary sizes and grid, on four k-points
        dict(_case("polarization", (2, 2, 1), 52, 400, 120, 200.0, "bf16x4"), name="p0_solid221_nao52_mixed"),
        dict(_case("self_energy", (2, 2, 1), 52, 400, 120, 200.0, "bf16x4"), name="sigma_step_solid221_nao52_mixed"),
        # the same contractions in the default (FP64) precision: a 2x2x2 solid of the serving stream ...
        dict(_case("polarization", (2, 2, 2), 26, 104, 80, 100.0), name="p0_solid222_nao26_fp64"),
        # ... and a molecule with odd sizes
        dict(_case("self_energy", (1, 1, 1), 45, 180, 80, 100.0), name="sigma_step_molecule_nao45_fp64"),
        # the screened interaction: the largest molecule of the batched workload (few, large matrices) ...
        dict(_case("screened", (1, 1, 1), 120, 480, 80, 100.0), name="screened_molecule_naux480"),
        # ... and the 3x3x3 solid (many matrices of medium size)
        dict(_case("screened", (3, 3, 3), 26, 200, 100, 100.0), name="screened_solid333_naux200"),
        # the Dyson update of G, called once per iteration and about ten times in a search for mu
        dict(_case("dyson", (3, 3, 3), 26, 200, 100, 100.0, overlap=False), name="dyson_solid333_nao26"),
        # the static self-energy of each iteration
        dict(_case("static", (3, 3, 3), 26, 200, 100, 100.0, "bf16x4", packed=False), name="static_solid333_nao26"),
        # molecules of uneven size, odd ones among them, through one batch
        dict(_case("batch", (1, 1, 1), 120, 480, 80, 100.0, "bf16x4", naos="13,24,37,58,81,120"), name="batch_molecules_mixed"),
        # second order on a molecule of the batched workload's shape
        dict(_case("gf2", (1, 1, 1), 26, 104, 80, 100.0, "bf16x4"), name="gf2_molecule_nao26_mixed"),
    ]


MESHES = [(1, 1, 1), (2, 1, 1), (2, 2, 1), (3, 1, 1), (2, 2, 2), (3, 2, 1), (3, 3, 1), (3, 3, 3)]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _seconds(c):
    """A rough device time of a pass from the work of each unit (for the size of the drawn cases)."""
    w = _flops(c)
    return w["fp64"] / 0.8e12 + w["mixed"] / 30e12


def draw(rng):
    while True:
        kind = rng.choice(["sigma", "polarization", "self_energy", "screened", "dyson", "static", "batch", "gf2"])
        precision = rng.choice(["fp64", "bf16x4"])
        mesh = rng.choice(MESHES)
        nao = _log(rng, 8, 120)
        naux = rng.choice([4 * nao, 3 * nao + rng.randrange(2 * nao)])
        ntau = _log(rng, 24, 120)
        beta = rng.choice([50.0, 100.0, 200.0])
        if kind == "batch":
            naos = sorted(_log(rng, 10, 120) for _ in range(rng.randrange(2, 9)))
            c = _case(kind, (1, 1, 1), naos[-1], 4 * naos[-1], ntau, beta, precision, naos=",".join(map(str, naos)))
        elif kind == "gf2":
            nao = _log(rng, 8, 40)
            c = _case(kind, (1, 1, 1), nao, 4 * nao, ntau, beta, precision)
        elif kind == "dyson":
            c = _case(kind, mesh, nao, 4 * nao, ntau, beta, precision, overlap=rng.random() < 0.3)
        elif kind == "static":
            c = _case(kind, mesh, nao, naux, ntau, beta, precision, packed=rng.random() < 0.3)
        else:
            c = _case(kind, mesh, nao, naux, ntau, beta, precision)
        if _seconds(c) <= 0.5 and _bytes_held(c) <= 24e9:
            return c


# ---- sizes ----------------------------------------------------------------------------------


def _nk(c):
    return c["n1"] * c["n2"] * c["n3"]


def _mesh(c):
    return (c["n1"], c["n2"], c["n3"])


def _systems(c):
    """(nao, naux) of every system of the case."""
    if c["kind"] == "batch":
        return [(int(x), 4 * int(x)) for x in c["naos"].split(",")]
    return [(c["nao"], c["naux"])]


def _nw(ntau, stat):
    return ntau if (ntau % 2 == 1) == (stat == 0) else ntau + 1


def _bytes_held(c):
    """Device bytes of a state, roughly: V, and the P arrays of the contexts that hold them."""
    nk, T, t = _nk(c), c["ntau"], 0
    for nao, naux in _systems(c):
        t += 16 * (2.5 * nk * nk * naux * nao * nao + 5 * nk * T * naux * naux)
    return t


def _flops(c):
    """Flops a pass cannot do without, by the unit that carries them."""
    nk, T, kind = _nk(c), c["ntau"], c["kind"]
    nw = _nw(T, 0)
    fp64 = mixed = 0.0
    for nao, naux in _systems(c):
        vgv = 8.0 * nk * nk * T * (2.0 * naux * nao ** 3 + naux ** 2 * nao ** 2)
        half = 0.5 if kind in ("sigma", "batch", "polarization", "gf2") else 1.0   # P0^q(beta - tau) = P0^-q(tau)^T
        contract = (half * vgv if kind in ("sigma", "batch", "polarization", "gf2") else 0.0) + \
                   (vgv if kind in ("sigma", "batch", "self_energy", "gf2") else 0.0)
        if kind in ("sigma", "batch", "screened"):
            h = 1.0 if kind == "screened" else 0.5
            fp64 += h * nk * (2 * 8.0 * T * nw * naux ** 2 + 8.0 * nw * naux ** 3)
        if kind == "dyson":
            fp64 += nk * (2 * 8.0 * T * nw * nao ** 2 + 8.0 * nw * nao ** 3)
        if kind == "static":
            fp64 += 16.0 * nk * nk * naux * nao ** 3
        if kind == "gf2":
            contract += 8.0 * T * (3.0 * naux * nao ** 3 + 2.0 * naux * nao ** 4 + nao ** 5)
        if c["precision"] == "fp64":
            fp64 += contract
        else:
            mixed += contract
    return {"fp64": fp64, "mixed": mixed}


def work(case):
    nk, T, kind = _nk(case), case["ntau"], case["kind"]
    w = _flops(case)
    n = 0.0
    for nao, naux in _systems(case):
        V, G, P = nk * nk * naux * nao ** 2, nk * T * nao ** 2, nk * T * naux ** 2
        n += {"sigma": V + 2 * G, "batch": V + 2 * G, "polarization": V + G + P, "self_energy": V + 2 * G + P,
              "screened": 2 * P, "dyson": 2 * G + nk * nao ** 2, "static": V * (0.5 if case.get("packed") else 1.0) + G,
              "gf2": V + 2 * G}[kind]
    return {"bytes": 16.0 * n, "flops": w["fp64"] + w["mixed"]}


# ---- inputs -----------------------------------------------------------------------------------


def _tau(ntau, beta):
    return 0.5 * beta * (1.0 - np.cos(np.pi * (np.arange(ntau) + 0.5) / ntau))


def _kpoints(mesh):
    return np.stack(np.meshgrid(*[np.arange(n) for n in mesh], indexing="ij"), -1).reshape(-1, 3)


def _shift(mesh, sign):
    """[k][q] -> flat index of k + sign q."""
    p, n = _kpoints(mesh), np.array(mesh)
    s = (p[:, None, :] + sign * p[None, :, :]) % n
    return (s[..., 0] * n[1] + s[..., 1]) * n[2] + s[..., 2]


def _unitary(n, rng):
    q, r = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    d = np.diagonal(r)
    return q * (d / np.abs(d))


def _hamiltonian(mesh, nao, rng):
    """H(k): eigenvalues in [-1.5, 1.5] Ha (molecule), or onsite [-0.75, 0.75] Ha plus hopping (solid)."""
    solid = mesh != (1, 1, 1)
    top = 0.75 if solid else 1.5
    u = _unitary(nao, rng)
    h0 = (u * rng.uniform(-top, top, nao)) @ u.conj().T
    hop = []
    for _ in range(3):
        x = rng.standard_normal((nao, nao)) + 1j * rng.standard_normal((nao, nao))
        x = 0.5 * (x + x.conj().T)
        hop.append(0.125 * x / np.linalg.norm(x, 2))
    kv = 2.0 * np.pi * _kpoints(mesh) / np.array(mesh)
    return np.stack([h0 + (sum(2.0 * np.cos(kv[k, d]) * hop[d] for d in range(3)) if solid else 0.0)
                     for k in range(len(kv))])


def _g_tau(h, beta, tau):
    """G0(k, tau) = -U e^{-e tau} / (1 + e^{-beta e}) U^dagger on the device."""
    e, u = np.linalg.eigh(h)
    a = np.abs(e)[:, None, :]
    s = np.where(e[:, None, :] >= 0, tau[None, :, None], beta - tau[None, :, None])
    f = torch.from_numpy(np.exp(-a * s) / (1.0 + np.exp(-beta * a))).to(DEV)
    u = torch.from_numpy(u).to(DEV)
    return -((u[:, None] * f[:, :, None, :]) @ u.conj().transpose(1, 2)[:, None]).contiguous()


def _gauss(shape, gen):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), dtype=torch.float64, device=DEV, generator=gen)) / math.sqrt(2.0)


def _decay(mesh, naux):
    return 40.0 if mesh != (1, 1, 1) else naux / 4.0


def _coulomb(mesh, nao, naux, gen):
    """V[k1][k2][Q][i][j], V^{k2 k1}_ji(Q) = conj V^{k1 k2}_ij(Q), amplitude exp(-Q / decay)."""
    nk = int(np.prod(mesh))
    c = torch.exp(-torch.arange(naux, dtype=torch.float64, device=DEV) / _decay(mesh, naux))[:, None, None]
    V = torch.empty((nk, nk, naux, nao, nao), dtype=C128, device=DEV)
    for a in range(nk):
        for b in range(a, nk):
            x = c * _gauss((naux, nao, nao), gen)
            if a == b:
                V[a, a] = 0.5 * (x + x.conj().transpose(1, 2))
            else:
                V[a, b] = x / math.sqrt(2.0)
                V[b, a] = V[a, b].conj().transpose(1, 2)
    return V


def _bosonic(mesh, naux, tau, beta, amp, gen):
    """A negative, decaying bosonic function with the symmetries of P0: Hermitian in QQ',
    X^q(beta - tau) = X^-q(tau)^T; X^q(tau) = -amp sum_m x_m x_m^dagger (e^{-d tau} + e^{-d (beta - tau)}) / (1 - e^{-d beta})."""
    nk = int(np.prod(mesh))
    minus = _shift(mesh, -1)[0]
    t = torch.from_numpy(tau).to(DEV)[:, None]
    d = 0.05 + 2.95 * torch.rand(naux, dtype=torch.float64, device=DEV, generator=gen)[None, :]
    f = amp / naux * (torch.exp(-d * t) + torch.exp(-d * (beta - t))) / (1.0 - torch.exp(-d * beta))
    c = torch.exp(-torch.arange(naux, dtype=torch.float64, device=DEV) / _decay(mesh, naux))[:, None]
    out = torch.empty((nk, len(tau), naux, naux), dtype=C128, device=DEV)
    for q in range(nk):
        p = int(minus[q])
        if p < q:
            out[q] = out[p].flip(0).transpose(1, 2)
            continue
        x = c * _gauss((naux, naux), gen)
        if p == q:
            x = x.real.to(C128)
        for k in range(len(tau)):
            out[q, k] = -(x * f[k]) @ x.conj().T
    return out


def _inputs(case, seed, nao, naux, salt=0):
    """The device arrays of one system, by name."""
    kind, mesh, T, beta = case["kind"], _mesh(case), case["ntau"], case["beta"]
    rng = np.random.default_rng([seed, salt])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed * 1009 + salt)
    tau = _tau(T, beta)
    x = {}
    if kind == "screened":
        x["P0t"] = _bosonic(mesh, naux, tau, beta, 7.0, gen)
        return x
    h = _hamiltonian(mesh, nao, rng)
    if kind == "dyson":
        x["H"] = torch.from_numpy(h).to(DEV)
        x["Sig"] = 0.05 * _g_tau(_hamiltonian(mesh, nao, rng), beta, tau)
        if case["overlap"]:
            us = [_unitary(nao, rng) for _ in range(_nk(case))]
            x["S"] = torch.from_numpy(np.stack([(u * rng.uniform(0.7, 1.3, nao)) @ u.conj().T for u in us])).to(DEV)
        return x
    x["G"] = _g_tau(h, beta, tau)
    x["V"] = _coulomb(mesh, nao, naux, gen)
    if kind == "self_energy":
        x["Pt"] = _bosonic(mesh, naux, tau, beta, 0.3, gen)
    return x


def prepare(case, seed):
    nk, T, kind = _nk(case), case["ntau"], case["kind"]
    state = {"kind": kind}
    if kind == "batch":
        systems = _systems(case)
        x = [_inputs(case, seed, nao, naux, i) for i, (nao, naux) in enumerate(systems)]
        cfgs = [gw.make_config(_mesh(case), nao, naux, T, case["beta"], spin_factor=SPIN, precision=case["precision"])
                for nao, naux in systems]
        batch = gw.gw_batch(cfgs, hbm_budget=BATCH_BUDGET)
        batch.set_coulomb([s["V"] for s in x])
        state.update(batch=batch, G=[s["G"] for s in x], V=[s["V"] for s in x], out=[torch.empty_like(s["G"]) for s in x])
        return state
    nao, naux = case["nao"], case["naux"]
    x = _inputs(case, seed, nao, naux)
    packed = bool(case.get("packed"))
    ctx = gw.gw_create(_mesh(case), nao, naux, T, case["beta"], mu=0.05, spin_factor=SPIN, precision=case["precision"],
                       v_packed=packed)
    shape = ctx.shapes()
    if "V" in x:
        if packed:
            x["V"] = torch.stack([x["V"][a, b] for a in range(nk) for b in range(a, nk)])
        gw.gw_set_coulomb(ctx, x["V"])
    if "S" in x:
        gw.gw_set_overlap(ctx, x["S"])
    out = {"polarization": shape["Pt"], "screened": shape["Pt"], "static": shape["H"]}.get(kind, shape["Sig"])
    state.update(x, ctx=ctx, out=torch.empty(out, dtype=C128, device=DEV))
    return state


def run(state):
    kind, out = state["kind"], state["out"]
    if kind == "batch":
        state["batch"].sigma_eval(state["G"], out)
        return out
    ctx = state["ctx"]
    if kind == "sigma":
        gw.gw_sigma_eval(ctx, state["G"], out)
    elif kind == "polarization":
        gw.gw_polarization(ctx, state["G"], out)
    elif kind == "self_energy":
        gw.gw_self_energy(ctx, state["G"], state["Pt"], out)
    elif kind == "screened":
        gw.gw_screened_interaction(ctx, state["P0t"], out)
    elif kind == "dyson":
        gw.gw_dyson_G(ctx, state["H"], state["Sig"], out)
    elif kind == "static":
        gw.gw_sigma_inf(ctx, state["G"], out)
    else:
        gw.gw_gf2_self_energy(ctx, state["G"], out)
    return out


# ---- the same in plain torch, complex128 ------------------------------------------------------


def _indices(n, stat):
    """The n sampled Matsubara indices (symmetric; dense up to n/3, then uniform in 1/m)."""
    if n <= 5:
        return np.array(sorted(sorted(range(-n - 1, n + 1), key=lambda m: (abs(2 * m + stat), m < 0))[:n]))
    M = n // 3
    core = list(range(-M - stat, M + 1))
    K = (n - len(core)) // 2
    tail = [(2 * M * (2 * K + 3) + (2 * K + 3 - 2 * j)) // (2 * (2 * K + 3 - 2 * j)) for j in range(1, K + 1)]
    return np.array(sorted(core + tail + [-t - stat for t in tail]))


@functools.lru_cache(maxsize=16)
def _grid(ntau, beta, stat):
    """omega [nw], F [nw][ntau] (Fourier integrals of the Chebyshev interpolant), B = its left inverse."""
    w = (2 * _indices(_nw(ntau, stat), stat) + stat) * np.pi           # times 1 / beta
    x, l = -np.cos(np.pi * (np.arange(ntau) + 0.5) / ntau), np.arange(ntau)
    C = np.cos(np.outer(l, np.arccos(x))) * np.where(l == 0, 1.0, 2.0)[:, None] / ntau
    panels = int(np.ceil((np.abs(w).max() / 2.0 + ntau) / 2.0)) + 8
    edge = -np.cos(np.pi * np.arange(panels + 1) / panels)
    g, gw_ = np.polynomial.legendre.leggauss(24)
    half = 0.5 * np.diff(edge)
    xq = (half[:, None] * (g + 1.0) + edge[:-1, None]).ravel()
    wq = (half[:, None] * gw_).ravel()
    Tnl = 0.5 * (np.exp(0.5j * np.outer(w, xq + 1.0)) * wq) @ np.cos(np.outer(np.arccos(np.clip(xq, -1, 1)), l))
    F = Tnl @ C
    B = np.linalg.pinv(F, rcond=1e-14)
    dev = lambda a: torch.from_numpy(a).to(DEV)                          # noqa: E731
    return w / beta, dev(F * beta), dev(B / beta)


def _along(M, X):
    """M [a][b] applied to axis 1 of X [n][b][...]."""
    n, b = X.shape[:2]
    return (M @ X.reshape(n, b, -1)).reshape((n, M.shape[0]) + tuple(X.shape[2:]))


def _p0(mesh, V, G):
    nk, T, nao, naux = G.shape[0], G.shape[1], G.shape[2], V.shape[2]
    kp = _shift(mesh, +1)
    P = torch.zeros((nk, T, naux, naux), dtype=C128, device=DEV)
    for q in range(nk):
        for k in range(nk):
            p = int(kp[k, q])
            for t in range(T):
                A = (V[k, p] @ G[p, t]).reshape(naux, -1)                                     # [Q][(d b)]
                Bm = (V[p, k] @ G[k, T - 1 - t]).transpose(1, 2).reshape(naux, -1)            # [Q'][(d b)]
                P[q, t] -= (SPIN / nk) * (A @ Bm.T)
    return P


def _sigma(mesh, V, G, P):
    nk, T, nao, naux = G.shape[0], G.shape[1], G.shape[2], V.shape[2]
    km = _shift(mesh, -1)
    S = torch.zeros_like(G)
    for q in range(nk):
        for k in range(nk):
            m = int(km[k, q])
            vm = V[m, k].reshape(naux, -1)
            for t in range(T):
                R = (P[q, t] @ vm).reshape(naux * nao, nao)                                   # [(Q b)][j]
                Z = (V[k, m] @ G[m, t]).transpose(0, 1).reshape(nao, naux * nao)              # [i][(Q b)]
                S[k, t] -= (1.0 / nk) * (Z @ R)
    return S


def _screen(ntau, beta, P0t):
    _, F, B = _grid(ntau, beta, 0)
    out = torch.empty_like(P0t)
    eye = torch.eye(P0t.shape[-1], dtype=C128, device=DEV)
    for q in range(P0t.shape[0]):
        Pw = _along(F, P0t[q:q + 1])[0]
        out[q] = _along(B, torch.linalg.solve(eye - Pw, Pw)[None])[0]
    return out


def _density(beta, G):
    T = G.shape[1]
    l, x = np.arange(T), -np.cos(np.pi * (np.arange(T) + 0.5) / T)
    w = (np.cos(np.outer(l, np.arccos(x))) * np.where(l == 0, 1.0, 2.0)[:, None] / T).sum(0)   # T_l(1) = 1
    return -torch.einsum("t,ktij->kij", torch.from_numpy(w).to(DEV).to(C128), G)


def _sigma_inf(beta, V, G):
    nk, naux, nao = V.shape[0], V.shape[2], V.shape[3]
    gam = _density(beta, G)
    rho = sum(torch.einsum("ab,Qba->Q", gam[k], V[k, k]) for k in range(nk))
    out = torch.empty_like(gam)
    for k in range(nk):
        out[k] = (SPIN / nk) * torch.einsum("Q,Qij->ij", rho, V[k, k])
        for p in range(nk):
            X = (V[k, p] @ gam[p]).transpose(0, 1).reshape(nao, -1)
            out[k] -= (1.0 / nk) * (X @ V[p, k].reshape(naux * nao, nao))
    return out


def _gf2(V, G):
    T, nao = G.shape[1], G.shape[2]
    S = _sigma((1, 1, 1), V, G, _p0((1, 1, 1), V, G))
    v = V[0, 0]
    n2 = nao * nao
    vr = v.reshape(-1, n2)
    for t in range(T):
        A = (v @ G[0, t]).reshape(-1, n2)
        D = (v @ G[0, T - 1 - t]).reshape(-1, n2)
        Y = (A.T @ A).reshape(nao, nao * n2)                       # [i][(q m l)]
        W = (D.T @ vr).reshape(nao * n2, nao)                      # [(q m l)][j]
        S[0, t] -= Y @ W
    return S


def exact(case, seed):
    kind, T, beta, mesh = case["kind"], case["ntau"], case["beta"], _mesh(case)
    # at about 1 TFLOP/s in complex128; a call per (q, k, tau) takes a few launches
    w = _flops(dict(case, precision="fp64"))
    calls = _nk(case) ** 2 * T if kind in ("sigma", "polarization", "self_energy") else T * len(_systems(case))
    if 2.0 * w["fp64"] / 0.9e12 + 2e-4 * calls > 18.0:
        return None
    one = lambda x: _sigma(mesh, x["V"], x["G"], _screen(T, beta, _p0(mesh, x["V"], x["G"])))   # noqa: E731
    if kind == "batch":
        return [one(_inputs(case, seed, nao, naux, i)) for i, (nao, naux) in enumerate(_systems(case))]
    x = _inputs(case, seed, case["nao"], case["naux"])
    if kind == "sigma":
        return one(x)
    if kind == "polarization":
        return _p0(mesh, x["V"], x["G"])
    if kind == "self_energy":
        return _sigma(mesh, x["V"], x["G"], x["Pt"])
    if kind == "screened":
        return _screen(T, beta, x["P0t"])
    if kind == "static":
        return _sigma_inf(beta, x["V"], x["G"])
    if kind == "gf2":
        return _gf2(x["V"], x["G"])
    wf, F, B = _grid(T, beta, 1)
    S = x["S"] if "S" in x else torch.eye(case["nao"], dtype=C128, device=DEV).expand_as(x["H"])
    z = torch.from_numpy(1j * wf + 0.05).to(DEV)[None, :, None, None]
    Gw = torch.linalg.inv(z * S[:, None] - x["H"][:, None] - _along(F, x["Sig"]))
    return _along(B, Gw)
