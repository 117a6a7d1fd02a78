"""What a user of the exchange library has it do, as cases that can be timed.

A case is one call (or the short run of calls that belongs together) through
the public entry points of paper_2207_04636_gb300, on a seeded periodic cell:
jittered atoms on a cubic lattice, periodised s/p/d Gaussians, S-orthonormal
occupied coefficients, interpolation points drawn from the basis density, and
auxiliary tables of translated Gaussian fitting functions, whose potentials
follow from one FFT (the "isdf" and "points" cases, which form or choose those
themselves, take pivoted points of the same basis).  Inputs are made with
torch on the GPU and handed over as a user's program has them: host arrays for
the blocking calls, device tensors for the enqueueing ones.
"""
import math

import torch

import paper_2207_04636_gb300 as xk

SPACING = 3.37  # bohr between lattice sites, as in the cubic benchmark cells


def listed():
    return [
        # the smallest SCF cells: launches and latency count
        {"name": "build 8 centres", "kind": "build", "mode": "f16x3", "centres": 8, "N": 104,
         "n": 16, "grid": 30, "naux": 520},
        # an ordinary member of a mixed-size workload (n <= 64)
        {"name": "build 27 centres", "kind": "build", "mode": "f16x3", "centres": 27, "N": 351,
         "n": 54, "grid": 45, "naux": 1755},
        # the headline workload: every SCF iteration of the 64-centre cell
        {"name": "build 64 centres", "kind": "build", "mode": "f16x3", "centres": 64, "N": 832,
         "n": 128, "grid": 60, "naux": 4000},
        # many occupied orbitals (n > 128: stored pair products)
        {"name": "build 27 centres n=200", "kind": "build", "mode": "f16x3", "centres": 27,
         "N": 351, "n": 200, "grid": 45, "naux": 1755},
        # a convergence check between full builds, ragged n
        {"name": "energy 27 centres n=100", "kind": "energy", "mode": "f16x3", "centres": 27,
         "N": 351, "n": 100, "grid": 45, "naux": 1755},
        # one SCF iteration as a host program drives it: K, E_x, then the ACE vectors
        {"name": "scf step 27 centres", "kind": "scf", "mode": "f16x3", "centres": 27, "N": 351,
         "n": 54, "grid": 45, "naux": 1755},
        # the one full exchange matrix at the end of an SCF run
        {"name": "full K 27 centres", "kind": "full", "mode": "f16x3", "centres": 27, "N": 351,
         "n": 54, "grid": 45, "naux": 1755},
        # the double-precision build a user checks the tensor path against
        {"name": "fp64 build 27 centres", "kind": "build", "mode": "fp64", "centres": 27, "N": 351,
         "n": 54, "grid": 45, "naux": 1755},
        # the Coulomb matrix that goes with every exchange build
        {"name": "coulomb 27 centres", "kind": "coulomb", "mode": "fp64", "centres": 27, "N": 351,
         "n": 54, "grid": 45, "naux": 1755},
        # a new geometry: tables formed on the device, to the first K and E_x
        {"name": "isdf set-up 27 centres", "kind": "isdf", "mode": "fp64", "centres": 27, "N": 351,
         "n": 54, "grid": 45, "naux": 1053},
        # interpolation points of a small cell, all grid points as candidates
        {"name": "points 8 centres", "kind": "points", "centres": 8, "N": 32, "grid": 24,
         "m": 13824, "want": 256},
        # a batch of SCF runs of different sizes, one call for all
        {"name": "batch of 6", "kind": "batch", "mode": "f16x3", "small": 4, "large": 2,
         "centres": 27, "N": 351, "n": 54, "grid": 45, "naux": 1755},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cell_sizes(rng, lo, hi, c_lo=3.0, c_hi=5.0):
    """Sizes of a cell of lo..hi centres: odd ones as often as round ones."""
    centres = _log(rng, lo, hi)
    k = math.ceil(centres ** (1 / 3) - 1e-9)
    N = 13 * centres - rng.randrange(0, 13)
    n = max(2, 2 * centres - rng.randrange(0, max(1, centres // 2)))
    grid = 15 * k - rng.randrange(0, 2 * k)
    naux = int(N * rng.uniform(c_lo, c_hi))
    return {"centres": centres, "N": N, "n": n, "grid": grid, "naux": min(naux, grid ** 3 // 4)}


def draw(rng):
    kind = rng.choice(["build", "build", "build", "wide", "energy", "scf", "full", "fp64",
                       "coulomb", "isdf", "points", "batch"])
    if kind == "points":
        grid = rng.randrange(14, 25)
        N = rng.randrange(26, 66)
        return {"kind": "points", "centres": 8, "N": N, "grid": grid,
                "m": rng.randrange(grid ** 3 // 2, grid ** 3 + 1), "want": _log(rng, 60, 257)}
    if kind == "batch":
        c = _cell_sizes(rng, 9, 27)
        return {"kind": "batch", "mode": "f16x3", "small": rng.randrange(1, 5),
                "large": rng.randrange(1, 3), **c}
    if kind == "wide":
        c = _cell_sizes(rng, 12, 27)
        c["n"] = min(c["N"], rng.randrange(129, 201))
        return {"kind": "build", "mode": "f16x3", **c}
    if kind == "build":
        return {"kind": "build", "mode": "f16x3", **_cell_sizes(rng, 4, 64, 3.0, 4.8)}
    if kind == "energy":
        c = _cell_sizes(rng, 4, 40)
        c["n"] = min(c["N"], c["n"] * rng.randrange(1, 3))
        return {"kind": "energy", "mode": "f16x3", **c}
    if kind == "isdf":
        return {"kind": "isdf", "mode": "fp64", **_cell_sizes(rng, 4, 27, 2.0, 3.0)}
    if kind in ("fp64", "coulomb"):
        return {"kind": "build" if kind == "fp64" else kind, "mode": "fp64",
                **_cell_sizes(rng, 4, 27, 2.0, 5.0)}
    return {"kind": kind, "mode": "f16x3", **_cell_sizes(rng, 4, 27)}


# ------------------------------------------------------------------ inputs

def _basis(case, g):
    """(Phi (N_g x N), L): periodised s, s, p, p, d Gaussians on jittered sites."""
    centres, N, grid = case["centres"], case["N"], case["grid"]
    k = math.ceil(centres ** (1 / 3) - 1e-9)
    L = SPACING * k
    dev = "cuda"
    site = torch.arange(centres, dtype=torch.float64)
    frac = torch.stack([site // (k * k), (site // k) % k, site % k], 1)
    pos = (frac + 0.5) * SPACING + (torch.rand(centres, 3, generator=g, dtype=torch.float64) - 0.5) * 0.1
    lo = torch.tensor([0.20, 0.80, 0.28, 0.90, 0.50], dtype=torch.float64)
    expo = lo * (1.0 + 0.5 * torch.rand(5, generator=g, dtype=torch.float64))
    # functions of one centre: (shell, [(coefficient, kx, ky, kz), ...])
    s, p = [(1.0, 0, 0, 0)], [[(1.0, 1, 0, 0)], [(1.0, 0, 1, 0)], [(1.0, 0, 0, 1)]]
    d = [[(1.0, 1, 1, 0)], [(1.0, 0, 1, 1)], [(1.0, 1, 0, 1)], [(0.5, 2, 0, 0), (-0.5, 0, 2, 0)],
         [(2 / 12 ** 0.5, 0, 0, 2), (-1 / 12 ** 0.5, 2, 0, 0), (-1 / 12 ** 0.5, 0, 2, 0)]]
    funs = [(0, s), (1, s)] + [(2, t) for t in p] + [(3, t) for t in p] + [(4, t) for t in d]
    per = -(-N // centres)
    funs = (funs * -(-per // len(funs)))[:per]
    x = torch.arange(grid, dtype=torch.float64, device=dev) * (L / grid)
    # per axis, centre and shell: sum_t d^j exp(-a d^2), j = 0, 1, 2
    T = int(math.ceil(math.sqrt(math.log(1e18) / 0.2) / L)) + 1
    dx = x[None, None, :, None] - pos.to(dev)[:, :, None, None] + L * torch.arange(
        -T, T + 1, dtype=torch.float64, device=dev)  # centre, axis, x, image
    ax = []
    for a in expo.tolist():
        e = torch.exp(-a * dx * dx)
        ax.append(torch.stack([e.sum(-1), (dx * e).sum(-1), (dx * dx * e).sum(-1)]))
    ax = torch.stack(ax)  # shell, power, centre, axis, x
    cols = [(c, f) for c in range(centres) for f in range(per)][:N]
    phi = torch.zeros(grid, grid, grid, N, dtype=torch.float64, device=dev)
    for t in range(3):
        sel = [(m, c, funs[f][0], *funs[f][1][t]) for m, (c, f) in enumerate(cols) if len(funs[f][1]) > t]
        if not sel:
            continue
        m, c, sh, co, kx, ky, kz = (torch.tensor(v, device=dev) for v in zip(*sel))
        fx, fy, fz = ax[sh, kx, c, 0], ax[sh, ky, c, 1], ax[sh, kz, c, 2]  # term, x
        yz = (fy * co.double()[:, None])[:, :, None] * fz[:, None, :]
        for i in range(grid):
            phi[i][:, :, m] += (fx[:, i, None, None] * yz).permute(1, 2, 0)
    phi = phi.reshape(grid ** 3, N)
    dV = L ** 3 / grid ** 3
    phi /= torch.sqrt(dV * (phi * phi).sum(0))
    return phi, L


def _coefficients(phi, dV, n, g):
    """C with C^T S C = 1: the Cholesky frame of S times random orthonormal columns."""
    N = phi.shape[1]
    Lc = torch.linalg.cholesky(dV * (phi.T @ phi))
    Q, _ = torch.linalg.qr(torch.randn(N, n, generator=g, dtype=torch.float64).to(phi.device))
    return torch.linalg.solve_triangular(Lc.T, Q, upper=True).contiguous()


def _tables(idx, naux, grid, L, g):
    """V (N_aux x N_g) and W (N_aux x N_aux) of Gaussian fitting functions a_g exp(-4 r^2)
    centred on the interpolation points: one FFT, then translations.  The a_g let the
    functions add up to at most one at every point, as a fit of the density does."""
    dev = "cuda"
    x = torch.arange(grid, dtype=torch.float64, device=dev) * (L / grid)
    one = sum(torch.exp(-4.0 * (x + t * L) ** 2) for t in range(-3, 4))
    chi = one[:, None, None] * one[None, :, None] * one[None, None, :]
    f = 2 * math.pi * torch.fft.fftfreq(grid, d=L / grid, dtype=torch.float64, device=dev)
    g2 = f[:, None, None] ** 2 + f[None, :, None] ** 2 + f[None, None, :] ** 2
    ker = torch.where(g2 > 0, 4 * math.pi / g2.clamp_min(1e-300), torch.zeros_like(g2))
    ck = torch.fft.fftn(chi)
    F = torch.fft.ifftn(ker * ck).real
    H = torch.fft.ifftn(ker * ck * ck.conj()).real
    amp = (0.5 + torch.rand(naux, generator=g, dtype=torch.float64)).to(dev)
    p = torch.stack([idx // (grid * grid), (idx // grid) % grid, idx % grid], 1)
    apart = tuple((p[:, None, :] - p[None, :, :]).remainder(grid).unbind(-1))
    amp = amp / (chi[apart] @ amp).max()
    W = H[apart] * amp[:, None] * amp
    W = 0.5 * (W + W.T)
    V = torch.empty(naux, grid, grid, grid, dtype=torch.float64, device=dev)
    r = torch.arange(grid, device=dev)
    for s in range(0, naux, 64):
        q = p[s:s + 64, :, None]
        i = (r - q).remainder(grid)
        V[s:s + 64] = F[i[:, 0, :, None, None], i[:, 1, None, :, None], i[:, 2, None, None, :]]
        V[s:s + 64] *= amp[s:s + 64, None, None, None]
    return V.reshape(naux, grid ** 3), W


def _pivots(rows, want):
    """Leading pivots of the pivoted Cholesky of (rows rows^T)^2, in plain torch."""
    X = (rows @ rows.T) ** 2
    d = X.diagonal().clone()
    Lc = torch.zeros(rows.shape[0], want, dtype=torch.float64, device=rows.device)
    piv = []
    for t in range(want):
        p = torch.argmax(d)[None]
        col = (X.index_select(1, p)[:, 0] - Lc[:, :t] @ Lc.index_select(0, p)[0, :t])
        Lc[:, t] = col / torch.sqrt(d.index_select(0, p))
        d = d - Lc[:, t] ** 2
        d.index_fill_(0, p, -1.0)
        piv.append(p)
    return torch.cat(piv)


def _cell(case, seed):
    """Every input of one cell as torch tensors on the GPU."""
    g = torch.Generator().manual_seed(1000003 * seed + 17)
    phi, L = _basis(case, g)
    grid, n, naux = case["grid"], case["n"], case["naux"]
    dV = L ** 3 / grid ** 3
    cell = {"phi": phi, "L": L, "dV": dV, "C": _coefficients(phi, dV, n, g)}
    # interpolation points sit where the basis does
    u = torch.rand(grid ** 3, generator=g, dtype=torch.float64).to(phi.device)
    key = torch.log(u) / (phi * phi).sum(1)  # weighted sampling without replacement
    if case["kind"] == "isdf":
        pool = torch.topk(key, min(grid ** 3, 3 * naux)).indices.sort().values
        cell["idx"] = pool[_pivots(phi[pool], naux)].sort().values
    else:
        cell["idx"] = torch.topk(key, naux).indices.sort().values
        cell["V"], cell["W"] = _tables(cell["idx"], naux, grid, L, g)
    return cell


def _members(case):
    """The cells of a batch: the case's own and the 8-centre one, several times each."""
    small = {"centres": 8, "N": 104, "n": 16, "grid": 30, "naux": 520, "kind": "build"}
    return [dict(small) for _ in range(case["small"])] + [
        dict(case, kind="build") for _ in range(case["large"])]


def _point_rows(case, seed):
    g = torch.Generator().manual_seed(1000003 * seed + 17)
    phi, _ = _basis(case, g)
    keep = torch.randperm(phi.shape[0], generator=g)[:case["m"]].sort().values
    return phi[keep.to(phi.device)].contiguous()


def _np(t):
    return t.cpu().numpy()


def _handle(case, c):
    """The handle of a geometry, as a user's program sets it up once."""
    return xk.Handle(_np(c["phi"]), _np(c["idx"]), _np(c["V"]), _np(c["W"]), c["dV"], case["n"],
                     mode=case["mode"])


# ----------------------------------------------------------------- running

def prepare(case, seed):
    kind = case["kind"]
    if kind == "points":
        return {"kind": kind, "rows": _np(_point_rows(case, seed)), "want": case["want"]}
    if kind == "batch":
        handles, Cs = [], []
        for k, m in enumerate(_members(case)):
            c = _cell(m, 64 * seed + k)
            handles.append(_handle(dict(m, mode=case["mode"]), c))
            Cs.append(_np(c["C"]))
        return {"kind": kind, "batch": xk.Batch(handles), "C": Cs}
    c = _cell(case, seed)
    st = {"kind": kind, "case": dict(case), "L": c["L"]}
    if kind == "isdf":
        st.update(phi=_np(c["phi"]), idx=_np(c["idx"]), C=_np(c["C"]))
        return st
    st["h"] = _handle(case, c)
    if kind in ("build", "energy"):
        st.update(C=c["C"], K=torch.empty_like(c["C"]),
                  Ex=torch.empty(1, dtype=torch.float64, device="cuda"))
    else:
        st["C"] = _np(c["C"])
    return st


def run(st):
    kind = st["kind"]
    if kind == "build":  # device in, device out, on the caller's stream
        st["h"].build_device(st["C"].data_ptr(), st["K"].data_ptr(), st["Ex"].data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
        return {"K": st["K"], "Ex": st["Ex"]}
    if kind == "energy":
        st["h"].energy_device(st["C"].data_ptr(), st["Ex"].data_ptr(),
                              torch.cuda.current_stream().cuda_stream)
        return {"Ex": st["Ex"]}
    if kind == "scf":
        K, Ex = st["h"].build(st["C"])
        Kij, xi, sign, _ = st["h"].ace()
        return {"K": K, "Ex": Ex, "Kij": Kij, "xi": xi, "sign": sign}
    if kind == "full":
        return {"K": st["h"].build_full(st["C"])}
    if kind == "coulomb":
        J, EJ = st["h"].coulomb(st["C"], st["case"]["grid"], st["L"])
        return {"J": J, "EJ": EJ}
    if kind == "isdf":
        h = xk.Handle.isdf(st["phi"], st["idx"], st["case"]["grid"], st["L"], st["case"]["n"],
                           mode=st["case"]["mode"])
        W, _, _ = h.tables()
        K, Ex = h.build(st["C"])
        h.release()
        return {"W": W, "K": K, "Ex": Ex}
    if kind == "points":
        return {"pivots": xk.isdf_points(st["rows"], st["want"])}
    K, Ex = st["batch"].build(st["C"])
    return {"K": K, "Ex": Ex}


# -------------------------------------------------------------------- work

def work(case):
    kind = case["kind"]
    if kind == "points":
        m, N, want = case["m"], case["N"], case["want"]
        return {"bytes": 8 * m * N, "flops": 2 * m * want * N + m * want * want}
    if kind == "batch":
        parts = [work(dict(m, mode=case["mode"])) for m in _members(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    N, n, na, ng = case["N"], case["n"], case["naux"], case["grid"] ** 3
    word = 8 if case["mode"] == "fp64" else 4  # the tables' type in the handle
    cell = {"bytes": word * (na * ng + na * na + ng * N) + 16 * N * n,
            "flops": 2 * ng * N * n + 6 * na * ng * n + 4 * na * na * n + 2 * n * N * (ng + 2 * na)}
    if kind == "energy":
        return {"bytes": cell["bytes"] - 8 * N * n,
                "flops": 2 * ng * N * n + 2 * na * ng * n + 2 * na * na * n}
    if kind == "full":
        return {"bytes": cell["bytes"] - 8 * N * n + 8 * N * N,
                "flops": 2 * ng * N * n + 2 * na * (ng + na) * (n + N) + 4 * na * N * N}
    if kind == "scf":
        return {"bytes": cell["bytes"] + 8 * (N * n + n * n + n),
                "flops": cell["flops"] + 2 * N * n * n + n ** 3 // 3 + N * n * n}
    if kind == "coulomb":
        return {"bytes": 8 * (ng * N + N * n + N * N), "flops": 2 * ng * N * (n + N) + 50 * ng}
    if kind == "isdf":
        fit = 2 * na * (ng + na) * N + na ** 3 // 3 + 2 * na * na * ng + 2 * na * na * ng
        return {"bytes": 8 * (ng * N + N * n + na * na + N * n),
                "flops": cell["flops"] + fit + 10 * na * ng * 16}
    return cell


# ------------------------------------------------------- 64-bit references

def _pois(f, grid, L):
    q = 2 * math.pi * torch.fft.fftfreq(grid, d=L / grid, dtype=torch.float64, device=f.device)
    g2 = q[:, None, None] ** 2 + q[None, :, None] ** 2 + q[None, None, :] ** 2
    ker = torch.where(g2 > 0, 4 * math.pi / g2.clamp_min(1e-300), torch.zeros_like(g2))
    out = torch.empty_like(f)
    for s in range(0, f.shape[0], 32):
        x = torch.fft.fftn(f[s:s + 32].reshape(-1, grid, grid, grid), dim=(1, 2, 3))
        out[s:s + 32] = torch.fft.ifftn(x * ker, dim=(1, 2, 3)).real.reshape(-1, grid ** 3)
    return out


def _exchange(c, full=False, energy_only=False):
    """K_{mu i} (or K_{mu nu}) and E_x of the robust pseudospectral exchange."""
    phi, C, idx, V, W, dV = c["phi"], c["C"], c["idx"], c["V"], c["W"], c["dV"]
    psi = phi @ C
    psig, phig = psi[idx], phi[idx]
    X, Xg, Y, Yg = (phig, phig, phi, phi) if full else (psig, phig, psi, phi)
    Q = psig @ psig.T
    ea = torch.zeros((), dtype=torch.float64, device=phi.device)
    M1 = torch.zeros(X.shape[1], phi.shape[0], dtype=torch.float64, device=phi.device)
    M2 = torch.empty(idx.numel(), Y.shape[1], dtype=torch.float64, device=phi.device)
    for s in range(0, idx.numel(), 512):
        P = psig[s:s + 512] @ psi.T
        V2 = V[s:s + 512] * P
        if energy_only:
            ea += (V2 * P).sum()
            continue
        M1 += X[s:s + 512].T @ V2
        M2[s:s + 512] = V2 @ Y
    if energy_only:
        return None, -dV * (2 * ea - (W * Q * Q).sum())
    lines = M1 @ Yg + M2.T @ Xg - ((W * Q) @ X).T @ Xg
    K = (dV * lines) if full else (dV * lines).T.contiguous()
    return K, None if full else -(K * C).sum()


def exact(case, seed):
    kind = case["kind"]
    if kind == "points":
        return None
    if kind == "batch":
        got = [_exchange(_cell(m, 64 * seed + k)) for k, m in enumerate(_members(case))]
        return {"K": [K.cpu() for K, _ in got], "Ex": [float(E) for _, E in got]}
    c = _cell(case, seed)
    if kind == "coulomb":
        psi = c["phi"] @ c["C"]
        rho = (psi * psi).sum(1)
        v = _pois(rho[None], case["grid"], c["L"])[0]
        J = c["dV"] * (c["phi"].T @ (v[:, None] * c["phi"]))
        return {"J": J.cpu(), "EJ": float(c["dV"] * (rho * v).sum())}
    if kind == "isdf":
        phig = c["phi"][c["idx"]]
        chi = torch.cholesky_solve((phig @ c["phi"].T) ** 2, torch.linalg.cholesky((phig @ phig.T) ** 2))
        c["V"] = _pois(chi, case["grid"], c["L"])
        W = c["V"] @ chi.T
        c["W"] = 0.5 * (W + W.T)
        K, E = _exchange(c)
        return {"W": c["W"].cpu(), "K": K.cpu(), "Ex": float(E)}
    if kind == "energy":
        return {"Ex": _exchange(c, energy_only=True)[1].reshape(1)}
    if kind == "full":
        return {"K": _exchange(c, full=True)[0].cpu()}
    K, E = _exchange(c)
    if kind == "scf":
        Kij = c["C"].T @ K
        Kij = 0.5 * (Kij + Kij.T)
        Lf = torch.linalg.cholesky(Kij)
        xi = torch.linalg.solve_triangular(Lf, K.T, upper=False).T
        return {"K": K.cpu(), "Ex": float(E), "Kij": Kij.cpu(), "xi": xi.contiguous().cpu(),
                "sign": torch.ones(case["n"], dtype=torch.float64)}
    return {"K": K, "Ex": E.reshape(1)}
