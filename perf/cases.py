"""Timed cases: the calls a user of the ISDF library makes, at the sizes the library is used at.

Each case names a public entry point (or the usual chain of them) and a size:

  gemm      the FP64-accurate tensor-core product, C = A B^T            (isdf_gemm_f64)
  rfft3     a batch of 3-D half spectra                                 (isdf_rfft3)
  select    interpolation points of a diamond cell                      (isdf_select_points)
  factor    fit and Coulomb matrix for given points: X^L, X^N, V        (isdf_fit, isdf_coulomb, isdf_get)
  build     the same and the first exchange build: K and E_x            (isdf_fit, isdf_coulomb, isdf_exchange)
  exchange  one exchange build of an SCF iteration: K or K C, and E_x   (isdf_exchange, isdf_exchange_occ)
  whole     a cell from its geometry to K and E_x                       (isdf_plan to isdf_exchange)

The cells are the displaced diamond supercells of paper_2404_09373_gb300/systems.py (13 functions
per atom, three grid levels, N_ip a few times N, two occupied orbitals per atom).  `exact` restates
each result in plain FP64 torch on the same inputs.

N_ip / N: the selection runs up to the benchmark's 6.  V itself is asked for up to 3 and K up to 5:
the condition number of C C^T grows steeply with the ratio, and above these the last digits of V
(of K) are set by the order of the FP64 operations in the Cholesky factorisation alone.
"""
import math

import numpy as np
import torch

from paper_2404_09373_gb300 import isdf as B
from paper_2404_09373_gb300 import systems as S

# the configuration of the library's benchmark: tensor-core products, exact prefilter, speculative blocks
TENSOR = {"precision": 1, "prefilter": 1, "select_block": 96}


def _cell(name, kind, reps, grid, ratio, **more):
    """reps: conventional cells per axis; grid: finest points per conventional cell edge (the
    coarser levels have a half and a quarter); ratio: N_ip / N."""
    return dict(name=name, kind=kind, rx=reps[0], ry=reps[1], rz=reps[2], grid=grid, ratio=ratio, **more)


def listed():
    return [
        # smallest call: one product of the sizes a single cell brings to the triangular inverse or
        # the W transform; dominated by launches and allocations
        dict(name="gemm_small", kind="gemm", M=391, N=208, K=208, digits=8),
        # the fit's shape: grid points x pivots x basis functions, 5 digits
        dict(name="gemm_fit", kind="gemm", M=131072, N=1824, K=832, digits=5),
        # the selection's shape: candidates x speculative set x basis functions, FP64 grade, ragged
        dict(name="gemm_columns", kind="gemm", M=250001, N=95, K=607, digits=8),
        # the spectra of some interpolation vectors on the finest grid of the 2x2x2 cell
        dict(name="rfft3_96", kind="rfft3", nx=96, ny=96, nz=96, batch=96),
        # points of one conventional cell (batched small cells, training cells of the proposer)
        _cell("select_cell", "select", (1, 1, 1), 48, 6.0),
        # points of the benchmark's supercell
        _cell("select_super", "select", (2, 2, 2), 48, 6.0),
        # the factors of a small supercell as a program takes them out: X^L, X^N and V
        _cell("factor_cell", "factor", (1, 1, 2), 48, 3.0),
        # points in hand to the first K: fit, Coulomb matrix and exchange of the benchmark's cell
        _cell("build_super", "build", (2, 2, 2), 48, 5.0),
        # the part of every SCF iteration: K of the benchmark's cell; K C (occ-RI) of a smaller one
        _cell("exchange_super", "exchange", (2, 2, 2), 48, 5.0, occ=False),
        _cell("exchange_occ", "exchange", (1, 2, 2), 48, 5.0, occ=True),
        # a whole small cell with the library's default options (plain FP64, step by step)
        _cell("whole_default", "whole", (1, 1, 1), 24, 3.0, tensor=False),
        # a whole cell in the benchmark's configuration, geometry to K
        _cell("whole_cell", "whole", (1, 1, 1), 48, 5.0, tensor=True),
    ]


_REPS = ((1, 1, 1), (1, 1, 2), (1, 2, 1), (2, 1, 1), (1, 2, 2), (2, 1, 2), (2, 2, 1), (1, 1, 3), (2, 2, 2))
# 40 and 3 x 48 points per axis are outside the double-float transform's sizes (cuFFT takes those)
_GRIDS = (24, 32, 40, 48)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("gemm", "gemm", "rfft3", "select", "factor", "build", "exchange", "exchange", "whole"))
    if kind == "gemm":
        c = dict(kind=kind, M=_log(rng, 64, 262144), N=_log(rng, 16, 2048), K=_log(rng, 32, 1024),
                 digits=rng.choice((5, 6, 7, 8)))
        while 2.0 * c["M"] * c["N"] * c["K"] > 4e11:
            c["M"] = c["M"] // 2 + 1
        return c
    if kind == "rfft3":
        n = [rng.choice((12, 16, 18, 24, 27, 32, 36, 48, 54, 64, 72, 81, 96, 108, 128)) for _ in range(3)]
        per = n[0] * n[1] * n[2]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], batch=max(1, min(_log(rng, 1, 2000), 85000000 // per)))
    ratio = round(rng.uniform(2.0, {"select": 6.0, "factor": 3.0}.get(kind, 5.0)), 3)
    grid = rng.choice(_GRIDS)
    if kind == "whole":
        tensor = rng.random() < 0.7
        reps = rng.choice(_REPS[:7] if tensor else _REPS[:1])
        if not tensor:
            grid, ratio = rng.choice((24, 32)), min(ratio, 4.0)
        c = _cell("", kind, reps, grid, ratio, tensor=tensor)
    elif kind == "exchange":
        c = _cell("", kind, rng.choice(_REPS), grid, ratio, occ=rng.random() < 0.5)
    else:
        c = _cell("", kind, rng.choice(_REPS), grid, ratio)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs


def _system(case, seed):
    rng = np.random.default_rng(S.SEED_BASE + 7919 * seed)
    g = case["grid"]
    grids = tuple((q, q, q) for q in (g, g // 2, g // 4))
    return S.make_system((case["rx"], case["ry"], case["rz"]), 0.05, rng, grids, S.LEVEL_EDGES_3), rng


def _nip(case, system):
    return int(case["ratio"] * S.nbasis(system))


def _functions(system):
    """Per basis function (shell order, a p shell's x, y, z): atom, exponent, powers, norm."""
    atom, alpha, pw = [], [], []
    for a, l, e in zip(system["shell_atom"], system["shell_l"], system["shell_exp"]):
        for c in range(1 if l == 0 else 3):
            atom.append(int(a))
            alpha.append(float(e))
            pw.append([int(l == 1 and c == ax) for ax in range(3)])
    alpha, pw = np.array(alpha), np.array(pw)
    norm = (2.0 * alpha / math.pi) ** 0.75 * np.where(pw.sum(1) == 1, 2.0 * np.sqrt(alpha), 1.0)
    return np.array(atom), alpha, pw, norm


def _orbitals(system, rng):
    """Seeded occupied orbitals, orthonormal in the analytic overlap of the periodic basis (what
    systems.make_orbitals computes pair by pair, over whole matrices)."""
    atom, alpha, pw, norm = _functions(system)
    n_occ = 2 * system["xyz"].shape[0]
    C0 = torch.from_numpy(rng.standard_normal((len(atom), n_occ))).cuda()
    al = torch.from_numpy(alpha).cuda()
    p = al[:, None] + al[None, :]
    mu = al[:, None] * al[None, :] / p
    sm = torch.from_numpy(np.outer(norm, norm)).cuda()
    for ax in range(3):
        L = float(system["edges"][ax])
        A = torch.from_numpy(system["xyz"][atom, ax].copy()).cuda()
        l = torch.from_numpy(pw[:, ax].copy()).cuda().bool()
        tmax = int(math.ceil(math.sqrt(40.0 / (0.5 * float(alpha.min()))) / L)) + 1
        tot = torch.zeros_like(p)
        for t in range(-tmax, tmax + 1):
            Bt = A[None, :] + t * L
            d = A[:, None] - Bt
            E = torch.exp(-mu * d * d) * torch.sqrt(math.pi / p)
            P = (al[:, None] * A[:, None] + al[None, :] * Bt) / p
            pa, pb = P - A[:, None], P - Bt
            v = torch.where(l[:, None], pa, torch.ones_like(p)) * torch.where(l[None, :], pb, torch.ones_like(p))
            tot += E * (v + torch.where(l[:, None] & l[None, :], 0.5 / p, torch.zeros_like(p)))
        sm *= tot
    w, U = torch.linalg.eigh(C0.T @ sm @ C0)
    return (C0 @ (U * w ** -0.5) @ U.T).contiguous()


def _dense(case, seed):
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
    # rows of different magnitude, as basis values and factor rows have
    a = torch.randn(case["M"], case["K"], dtype=torch.float64, device="cuda", generator=g)
    a *= torch.exp(2.0 * torch.randn(case["M"], 1, dtype=torch.float64, device="cuda", generator=g))
    b = torch.randn(case["N"], case["K"], dtype=torch.float64, device="cuda", generator=g)
    return a, b


def _grid_batch(case, seed):
    """Functions localised like interpolation vectors: a few Gaussian products on the grid each."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 29)
    out = torch.zeros(case["batch"], case["nz"], case["ny"], case["nx"], dtype=torch.float64, device="cuda")
    r = torch.rand(4, 5, case["batch"], dtype=torch.float64, device="cuda", generator=g)
    for centre in r:
        f = [centre[4] * 2.0 - 0.5]
        for ax, n in enumerate((case["nz"], case["ny"], case["nx"])):
            u = torch.arange(n, dtype=torch.float64, device="cuda") / n
            d = u[None, :] - centre[ax][:, None]
            d = d - torch.round(d)
            f.append(torch.exp(-(20.0 + 200.0 * centre[3][:, None]) * d * d))
        out += torch.einsum("b,bz,by,bx->bzyx", *f)
    return out


def _plan(case, seed):
    system, rng = _system(case, seed)
    return system, rng, B.isdf_plan(system, TENSOR)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        a, b = _dense(case, seed)
        return dict(kind=kind, a=a, b=b, c=torch.empty(case["M"], case["N"], dtype=torch.float64, device="cuda"),
                    digits=case["digits"])
    if kind == "rfft3":
        f = _grid_batch(case, seed)
        s = torch.empty(case["batch"], case["nz"], case["ny"], case["nx"] // 2 + 1, dtype=torch.complex128, device="cuda")
        return dict(kind=kind, f=f, s=s)
    if kind == "whole":
        system, rng = _system(case, seed)
        C = _orbitals(system, rng)
        return dict(kind=kind, system=system, nip=_nip(case, system), C=C, options=TENSOR if case["tensor"] else None)
    system, rng, plan = _plan(case, seed)
    nip, nf = _nip(case, system), S.nbasis(system)
    state = dict(kind=kind, plan=plan, nip=nip)
    if kind == "select":
        return state
    piv, _ = B.isdf_select_points(plan, nip)
    state["piv"] = piv
    if kind == "build":
        state["C"] = _orbitals(system, rng)
        state["K"] = torch.empty((nf, nf), dtype=torch.float64, device="cuda")
        return state
    if kind == "factor":
        for k, shape in (("V", (nip, nip)), ("XL", (nf, nip)), ("XN", (nf, nip))):
            state[k] = torch.empty(shape, dtype=torch.float64, device="cuda")
        return state
    B.isdf_fit(plan, piv)
    B.isdf_coulomb(plan)
    B.isdf_release_fit(plan)
    state["C"] = _orbitals(system, rng)
    state["occ"] = case["occ"]
    state["K"] = torch.empty((nf, state["C"].shape[1] if case["occ"] else nf), dtype=torch.float64, device="cuda")
    return state


# ---------------------------------------------------------------- the timed pass


def run(s):
    kind = s["kind"]
    if kind == "gemm":
        return B.isdf_gemm_f64(s["a"], s["b"], s["c"], slices=s["digits"])
    if kind == "rfft3":
        return B.isdf_rfft3(s["f"], s["s"])
    if kind == "select":
        piv, dval = B.isdf_select_points(s["plan"], s["nip"])
        return {"pivots": piv, "dval": dval}
    if kind == "factor":
        B.isdf_fit(s["plan"], s["piv"])
        B.isdf_coulomb(s["plan"], s["V"])
        B.isdf_get(s["plan"], B.GET_XL, s["XL"])
        B.isdf_get(s["plan"], B.GET_XN, s["XN"])
        return {"V": s["V"], "XL": s["XL"], "XN": s["XN"]}
    if kind == "build":
        B.isdf_fit(s["plan"], s["piv"])
        B.isdf_coulomb(s["plan"])
        K, Ex = B.isdf_exchange(s["plan"], s["C"], s["K"])
        return {"K": K, "Ex": Ex}
    if kind == "exchange":
        K, Ex = (B.isdf_exchange_occ if s["occ"] else B.isdf_exchange)(s["plan"], s["C"], s["K"])
        return {"K": K, "Ex": Ex}
    plan = B.isdf_plan(s["system"], s["options"])
    try:
        piv, dval = B.isdf_select_points(plan, s["nip"])
        B.isdf_fit(plan, piv)
        B.isdf_coulomb(plan)
        K, Ex = B.isdf_exchange(plan, s["C"])
    finally:
        plan.close()
    return {"pivots": piv, "dval": dval, "K": K, "Ex": Ex}


# ---------------------------------------------------------------- work


def work(case):
    """Bytes of the inputs and outputs, and the FP64 operations of the method (one multiply-add = 2)."""
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 8.0 * (M * K + N * K + M * N), "flops": 2.0 * M * N * K}
    if kind == "rfft3":
        n = case["nx"] * case["ny"] * case["nz"]
        nq = (case["nx"] // 2 + 1) * case["ny"] * case["nz"]
        return {"bytes": case["batch"] * (8.0 * n + 16.0 * nq), "flops": case["batch"] * 2.5 * n * math.log2(n)}
    atoms = 8 * case["rx"] * case["ry"] * case["rz"]
    nf, n_occ = 13 * atoms, 2 * atoms
    nip = int(case["ratio"] * nf)
    cells = case["rx"] * case["ry"] * case["rz"]
    ng = [cells * q ** 3 for q in (case["grid"], case["grid"] // 2, case["grid"] // 4)]
    fL, fG = [5 * atoms, 4 * atoms, 4 * atoms], [13 * atoms, 8 * atoms, 4 * atoms]
    share = [0.39, 0.40, 0.21]  # of the pivots, per level, on these cells
    phi = 8.0 * sum(a * b for a, b in zip(fG, ng))
    out = {"bytes": 0.0, "flops": 0.0}
    if kind in ("select", "whole"):
        out["bytes"] += phi + 16.0 * nip
        # columns of M and of the factor at the candidates (about a third of the points)
        out["flops"] += sum(2.0 * h * nip * (n / 3.0) * (g + 0.5 * h * nip) for h, n, g in zip(share, ng, fG))
    if kind in ("factor", "build", "whole"):
        out["bytes"] += phi + 8.0 * nip * nip + 16.0 * nf * nip
        k = [h * nip for h in share]
        out["flops"] += sum(2.0 * q * n * g + q ** 3 + 5.0 * q * n * math.log2(n) for q, n, g in zip(k, ng, fG))
        out["flops"] += sum((1.0 if a == b else 2.0) * k[a] * k[b] * ng[b] for a in range(3) for b in range(a, 3))
    if kind in ("build", "exchange", "whole"):
        occ = case.get("occ", False)
        out["bytes"] += 8.0 * nip * nip + 16.0 * nf * nip + 8.0 * nf * n_occ + 8.0 * nf * (n_occ if occ else nf)
        out["flops"] += 4.0 * nip * nip * n_occ
        # W times the occupied projections, or times the nonzero blocks of [X^L X^N]
        cols = [4.0 * nip * n_occ] if occ else [f * h * nip for f, h in zip(fL, (0.39, 1.18, 1.79))]
        out["flops"] += sum(2.0 * 2.0 * nip * c for c in cols)
    return out


# ---------------------------------------------------------------- plain FP64


def _level_data(system):
    atom, alpha, pw, norm = _functions(system)
    edges = system["level_min_exp"]
    return atom, alpha, pw, norm, np.array([int(np.sum(edges > a)) for a in alpha])


def _phi(system, level):
    """Basis values of a level (its own functions, then the coarser ones) on its grid, and the set sizes."""
    atom, alpha, pw, norm, lev = _level_data(system)
    rows = np.concatenate([np.flatnonzero(lev == level), np.flatnonzero(lev > level)])
    nx, ny, nz = (int(q) for q in system["grids"][level])
    tabs = []
    for ax, n in enumerate((nx, ny, nz)):
        L = float(system["edges"][ax])
        x = np.arange(n) * (L / n)
        tab = np.zeros((rows.size, n))
        for i, f in enumerate(rows):
            A, a = float(system["xyz"][atom[f], ax]), float(alpha[f])
            rc = math.sqrt(math.log(1.0 / system["image_tol"]) / a)
            for t in range(-int((rc + L) / L) - 2, int((rc + L) / L) + 3):
                c = A + t * L
                if max(-c, c - L, 0.0) <= rc:
                    u = x - A - t * L
                    tab[i] += (u if pw[f, ax] else 1.0) * np.exp(-a * u * u)
        tabs.append(torch.from_numpy(tab).cuda())
    tabs[0] *= torch.from_numpy(norm[rows]).cuda()[:, None]
    phi = torch.empty(rows.size, nz * ny * nx, dtype=torch.float64, device="cuda")
    for i in range(rows.size):
        torch.mul((tabs[2][i][:, None] * tabs[1][i][None, :])[:, :, None], tabs[0][i], out=phi[i].view(nz, ny, nx))
    return phi, int(np.sum(lev == level)), rows


def _greedy(system, nip):
    """Pivots and pivot values of the greedy pivoted Cholesky over the points whose initial residual is
    at least 1e-6 of the largest (residuals never grow, so the others are never picked while the pivot
    values stay above that; None if they do not)."""
    omega = float(np.prod(system["edges"]))
    d, phis, tau = [], [], None
    for l, g in enumerate(system["grids"]):
        phi, nL, _ = _phi(system, l)
        w = omega / float(np.prod(g))
        aL, aN = phi[:nL].square().sum(0), phi[nL:].square().sum(0)
        d.append(w * aL * (aL + 2.0 * aN))
        phis.append((phi, nL, w))
    d0 = max(float(x.max()) for x in d)
    keep = [torch.nonzero(x >= 1e-6 * d0).ravel() for x in d]
    off = np.concatenate([[0], np.cumsum([k.numel() for k in keep])])
    lev = []
    for l, k in enumerate(keep):
        phi, nL, w = phis[l]
        phis[l] = None
        lev.append((phi[:, k].contiguous(), nL, w, torch.empty(min(nip, k.numel()), k.numel(), dtype=torch.float64, device="cuda")))
        del phi
    d = torch.cat([x[k] for x, k in zip(d, keep)])
    piv, dval, ncol = [], [], [0] * len(keep)
    for _ in range(nip):
        top = float(d.max())
        p = int(torch.argmax((d >= top - max(1e-9 * top, 1e-13 * d0)).to(torch.int8)))
        l = int(np.searchsorted(off, p, side="right")) - 1
        t = p - int(off[l])
        phi, nL, w, fac = lev[l]
        k = ncol[l]
        aL = phi[:nL, t] @ phi[:nL]
        aN = phi[nL:, t] @ phi[nL:]
        v = w * aL * (aL + 2.0 * aN)
        if k:
            v -= fac[:k, t] @ fac[:k]
        dp = float(d[p])
        v /= math.sqrt(dp)
        v[t] = math.sqrt(dp)
        fac[k] = v
        part = d[int(off[l]):int(off[l + 1])]
        part -= v * v
        part[t] = 0.0
        ncol[l] += 1
        piv.append((l << B.PIVOT_SHIFT) | int(keep[l][t]))
        dval.append(dp)
    if min(dval) < 2e-6 * d0:
        return None
    return np.array(piv, dtype=np.int64), np.array(dval)


def _vectors(system, piv):
    """Per level: Xi^T [k][ng]; and X^L, X^N over all pivots (level by level)."""
    lo = np.concatenate([piv[(piv >> B.PIVOT_SHIFT) == l] for l in range(len(system["grids"]))])
    nf, nip = S.nbasis(system), piv.size
    XL = torch.zeros(nf, nip, dtype=torch.float64, device="cuda")
    XN = torch.zeros_like(XL)
    xi, c0 = [], 0
    for l in range(len(system["grids"])):
        g = torch.from_numpy(lo[(lo >> B.PIVOT_SHIFT) == l] & ((1 << B.PIVOT_SHIFT) - 1)).cuda()
        phi, nL, rows = _phi(system, l)
        P = phi[:, g].contiguous()
        k = g.numel()
        XL[torch.from_numpy(rows[:nL]).cuda(), c0:c0 + k] = P[:nL]
        XN[torch.from_numpy(rows[nL:]).cuda(), c0:c0 + k] = P[nL:]
        c0 += k
        z = P[nL:].T @ phi[nL:]
        z *= 2.0
        a = P[:nL].T @ phi[:nL]
        z += a
        z *= a
        del a, phi
        cc = z[:, g]
        chol = torch.linalg.cholesky(0.5 * (cc + cc.T)) if k else cc
        for j in range(0, z.shape[1] if k else 0, 131072):
            z[:, j:j + 131072] = torch.cholesky_solve(z[:, j:j + 131072].contiguous(), chol)
        xi.append(z)
    return xi, XL, XN


def _coulomb(system, xi):
    omega, edges = float(np.prod(system["edges"])), system["edges"]
    nip = sum(x.shape[0] for x in xi)
    V = torch.zeros(nip, nip, dtype=torch.float64, device="cuda")
    off = np.concatenate([[0], np.cumsum([x.shape[0] for x in xi])])
    n = [tuple(int(q) for q in g) for g in system["grids"]]  # nx, ny, nz

    def half(a, b):
        """Spectra of level a's vectors on level b's modes (a mode at n/2 split evenly), q_x in [0, n/2]."""
        (fx, fy, fz), (cx, cy, cz), k = n[a], n[b], xi[a].shape[0]
        out = torch.empty(k, cz, cy, cx // 2 + 1, dtype=torch.complex128, device="cuda")
        for j in range(0, k, 64):
            f = xi[a][j:j + 64].view(-1, fz, fy, fx)
            if a == b:
                out[j:j + 64] = torch.fft.rfftn(f, dim=(1, 2, 3))
                continue
            s = torch.fft.fftn(f, dim=(1, 2, 3))
            for dim, nf, nc in ((1, fz, cz), (2, fy, cy), (3, fx, cx)):
                m = torch.cat([torch.arange(nc // 2 + 1), torch.arange(-(nc // 2) + 1, 0)]).cuda()
                u = s.index_select(dim, m % nf)
                u.select(dim, nc // 2).add_(s.select(dim, nf - nc // 2)).mul_(0.5)
                s = u
            out[j:j + 64] = s[..., :cx // 2 + 1]
        return out.view(k, -1)

    for b in range(len(xi)):
        if not xi[b].shape[0]:
            continue
        nx, ny, nz = n[b]
        q = [torch.arange(nx // 2 + 1).cuda(), torch.fft.fftfreq(ny, 1.0 / ny).cuda(), torch.fft.fftfreq(nz, 1.0 / nz).cuda()]
        G = [2.0 * math.pi * x.double() / float(e) for x, e in zip(q, edges)]
        G2 = G[2][:, None, None] ** 2 + G[1][None, :, None] ** 2 + G[0][None, None, :] ** 2
        w = torch.where(G2 > 0, 4.0 * math.pi * omega / torch.where(G2 > 0, G2, torch.ones_like(G2)), torch.zeros_like(G2))
        w[:, :, 1:nx // 2] *= 2.0
        ny2 = w.clone()
        ny2[:, :, nx // 2] *= 0.5
        ny2[:, ny // 2, :] *= 0.5
        ny2[nz // 2, :, :] *= 0.5
        sb = half(b, b)
        for a in range(b + 1):
            if not xi[a].shape[0]:
                continue
            sa = sb if a == b else half(a, b)
            wt = (ny2 if a == b else w).reshape(-1) / (float(np.prod(n[a])) * float(np.prod(n[b])))
            blk = torch.zeros(xi[a].shape[0], xi[b].shape[0], dtype=torch.float64, device="cuda")
            for j in range(0, sb.shape[1], 1 << 17):
                l = torch.view_as_real(sa[:, j:j + (1 << 17)] * wt[j:j + (1 << 17)]).flatten(1)
                blk += l @ torch.view_as_real(sb[:, j:j + (1 << 17)].contiguous()).flatten(1).T
            V[off[a]:off[a + 1], off[b]:off[b + 1]] = blk
            V[off[b]:off[b + 1], off[a]:off[a + 1]] = blk.T
            del sa
        del sb
    return V


def _exchange(V, XL, XN, C):
    yl, yn = XL.T @ C, XN.T @ C
    yg = yl + yn
    T = torch.cat([(V * (yg @ yg.T)) @ XL.T + (V * (yg @ yl.T)) @ XN.T,
                   (V * (yl @ yg.T)) @ XL.T + (V * (yl @ yl.T)) @ XN.T])
    K = torch.cat([XL, XN], 1) @ T
    KC = K @ C
    return K, KC, -float((C * KC).sum())


def exact(case, seed):
    """What run() returns for these inputs in plain FP64.  The points of the factor, build and exchange
    cases are inputs (prepare() selects them); the select and whole cases find theirs here."""
    kind = case["kind"]
    if kind == "gemm":
        a, b = _dense(case, seed)
        return a @ b.T
    if kind == "rfft3":
        return torch.fft.rfftn(_grid_batch(case, seed), dim=(1, 2, 3))
    system, rng = _system(case, seed)
    nip = _nip(case, system)
    if kind in ("select", "whole"):
        if case["rx"] * case["ry"] * case["rz"] > 4:
            return None
        found = _greedy(system, nip)
        if found is None:
            return None
        piv, dval = found
        if kind == "select":
            return {"pivots": None, "dval": dval}
    else:
        system, rng, plan = _plan(case, seed)
        piv, _ = B.isdf_select_points(plan, nip)
        plan.close()
    xi, XL, XN = _vectors(system, piv)
    V = _coulomb(system, xi)
    del xi
    if kind == "factor":
        return {"V": V, "XL": XL, "XN": XN}
    K, KC, Ex = _exchange(V, XL, XN, _orbitals(system, rng))
    if kind in ("build", "exchange"):
        return {"K": KC if case.get("occ", False) else K, "Ex": Ex}
    return {"pivots": None, "dval": dval, "K": K, "Ex": Ex}
