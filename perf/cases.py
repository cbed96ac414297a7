"""What the speed of this framework is measured on: passes through its public entry points.

The cases are the steps of a GW run (polarization, screened interaction, correlation
self-energy, analytic continuation) as a program calls them, from the smallest system, where
the launches count, to the sizes of the 4x4x4-mesh benchmark workload. Inputs are drawn on the
device from the seed with the laws of the repository's synthetic workloads: projections
(N(0,1) + i N(0,1)) / (1 + I/16), occupied energies U[-0.5, 0] Ha, unoccupied U[0.05, 2] Ha, a
k+q permutation of the mesh, Coulomb eigenvalues 4 pi / (0.1 + I^(2/3)), tan-mapped
Gauss-Legendre frequencies up to 50 Ha. Output buffers and workspaces of the large calls are
laid out once in prepare(), as the benchmark's own pipeline keeps them.
"""
import math
import random

import numpy as np
import torch

import paper_1003_0316_gb300 as gw

MSIG_SCALE = 2.0 ** -5         # self-energy projections of the mesh workloads


def listed():
    return [
        # a whole small calculation (8 k points, 32 bands, 64 basis functions) with the default
        # precision: every call is short, so launches and host work count
        {"name": "chain_small_fp64", "kind": "chain", "precision": "fp64", "nk": 8, "nocc": 4,
         "nunocc": 28, "nb": 64, "nw": 8, "nq": 1},
        # the main step at the benchmark's size: two of its q points (K = 409,600 each)
        {"name": "polarization_bf16x3_mesh", "kind": "polarization", "precision": "bf16x3",
         "nq": 2, "nk": 64, "nocc": 16, "nunocc": 400, "nb": 600, "nw": 16, "real": False},
        # the more accurate split at a quarter of the k points of one such q
        {"name": "polarization_tf32x3_q", "kind": "polarization", "precision": "tf32x3",
         "nq": 1, "nk": 16, "nocc": 16, "nunocc": 400, "nb": 600, "nw": 16, "real": False},
        # q points of unequal, partly odd basis sizes and band counts in one call
        # (N_b of 300 to 1500, 200 to 800 unoccupied bands, 32 occupied)
        {"name": "polarization_bf16x3_uneven", "kind": "polarization", "precision": "bf16x3",
         "nq": 4, "nk": 8, "nocc": 32, "nunocc": 200, "nunocc_max": 800, "nb": 300,
         "nb_max": 1500, "nw": 16, "real": False},
        # a crystal with inversion symmetry: real projections, odd basis size, real solve
        {"name": "inversion_p_and_w", "kind": "real_pw", "precision": "bf16x3", "nq": 2,
         "nk": 8, "nocc": 16, "nunocc": 400, "nb": 333, "nw": 16},
        # the default (FP64) polarization at the benchmark's basis size, two frequencies
        {"name": "polarization_fp64_q", "kind": "polarization", "precision": "fp64", "nq": 1,
         "nk": 16, "nocc": 16, "nunocc": 400, "nb": 600, "nw": 2, "real": False},
        # the screened interaction of the benchmark's 8 q points at all 16 frequencies
        {"name": "screened_w_mesh", "kind": "screened_w", "nq": 8, "nb": 600, "nw": 16,
         "real": False},
        # the self-energy of 16 states over 416 bands and 8 q points, as the benchmark runs it
        {"name": "sigma_c_tf32x3_mesh", "kind": "sigma", "precision": "tf32x3", "nq": 8,
         "nstates": 16, "nbands": 416, "nb": 600, "nw": 16},
        # the same with the default (FP64) precision for one q point
        {"name": "sigma_c_fp64_q", "kind": "sigma", "precision": "fp64", "nq": 1,
         "nstates": 16, "nbands": 416, "nb": 600, "nw": 16},
        # the continuation of many curves (every band and k point of a data set)
        {"name": "fit_100k_curves", "kind": "fit", "n": 100000, "nw": 24, "npole": 2},
        # the continuation of one calculation's 16 states
        {"name": "fit_16_curves", "kind": "fit", "n": 16, "nw": 16, "npole": 2},
        # one training step of the learned start (backward and Adam)
        {"name": "mlp_train_step", "kind": "train", "batch": 512},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds: sizes over their whole ranges, odd ones among them."""
    kind = rng.choice(["chain", "polarization", "polarization", "polarization", "real_pw",
                       "screened_w", "screened_w", "sigma", "sigma", "fit"])
    if kind == "chain":
        return {"kind": kind, "precision": "fp64", "nk": rng.choice([1, 2, 4, 8]),
                "nocc": rng.randint(2, 8), "nunocc": rng.randint(9, 60), "nb": _log(rng, 24, 150),
                "nw": rng.randint(6, 16), "nq": rng.randint(1, 2)}
    if kind == "polarization":
        prec = rng.choice(["bf16x3", "bf16x3", "tf32x3", "fp64"])
        # the rows of a split-precision call (its error bounds are stated from about 1e5 rows
        # for BF16), far fewer for the FP64 pipe
        K = _log(rng, 2000, 40000) if prec == "fp64" else _log(rng, 20000, 120000)
        nk, nocc = rng.choice([4, 8, 16]), rng.randint(2, 16)
        return {"kind": kind, "precision": prec, "nq": rng.randint(1, 3), "nk": nk, "nocc": nocc,
                "nunocc": max(3, K // (nk * nocc)),
                "nb": _log(rng, 65, 500) if prec == "fp64" else _log(rng, 65, 900),
                "nw": rng.randint(1, 4) if prec == "fp64" else rng.randint(2, 20),
                "real": prec != "fp64" and rng.random() < 0.3}
    if kind == "real_pw":
        return {"kind": kind, "precision": rng.choice(["bf16x3", "tf32x3"]), "nq": rng.randint(1, 3),
                "nk": 8, "nocc": rng.randint(4, 16), "nunocc": rng.randint(100, 500),
                "nb": _log(rng, 65, 500), "nw": rng.randint(4, 16)}
    if kind == "screened_w":
        return {"kind": kind, "nq": rng.randint(1, 6), "nb": _log(rng, 48, 900),
                "nw": rng.randint(2, 16), "real": rng.random() < 0.4}
    if kind == "sigma":
        prec = rng.choice(["tf32x3", "bf16x3", "fp64"])
        return {"kind": kind, "precision": prec, "nq": rng.randint(1, 2 if prec == "fp64" else 6),
                "nstates": rng.randint(3, 16), "nbands": rng.randint(40, 300),
                "nb": _log(rng, 64, 400 if prec == "fp64" else 800), "nw": rng.randint(6, 20)}
    npole = rng.choice([1, 2, 2, 2, 3])
    return {"kind": "fit", "n": _log(rng, 12, 40000 if npole < 3 else 8000),
            "nw": rng.choice([12, 16, 20, 24, 33]), "npole": npole}


# ---------------------------------------------------------------- inputs
def _omega(nw, omega_max=50.0):
    x, _ = np.polynomial.legendre.leggauss(nw)
    return np.tan(0.5 * (x + 1.0) * np.arctan(omega_max))


def _coulomb(nb, dev):
    i = torch.arange(nb, dtype=torch.float64, device=dev)
    return 4.0 * math.pi / (0.1 + i ** (2.0 / 3.0))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _sizes(c):
    """(N_b, N_unocc) of every q: the same for all, or spread over the case's ranges."""
    if "nb_max" not in c:
        return [(c["nb"], c["nunocc"])] * c["nq"]
    r = random.Random(c["nb_max"] * 31 + c["nq"])
    return [(r.randint(c["nb"], c["nb_max"]), r.randint(c["nunocc"], c["nunocc_max"]))
            for _ in range(c["nq"])]


def _uniform(g, shape):
    return torch.rand(shape, generator=g, dtype=torch.float64, device="cuda")


def _projections(g, rows, nb, dtype, scale=1.0):
    decay = scale / (1.0 + torch.arange(nb, dtype=torch.float64, device="cuda") / 16.0)
    if dtype == torch.float32:
        return torch.randn((rows, nb), generator=g, device="cuda").mul_(decay.float())
    part = torch.float64 if dtype == torch.complex128 else torch.float32
    x = torch.randn((rows, nb, 2), generator=g, dtype=part, device="cuda")
    return torch.view_as_complex(x.mul_(decay.to(part)[:, None]))


def _polar_inputs(c, seed, real):
    """Per q: the projections [K][N_b] and the transition energies [K]."""
    g = _gen(seed)
    dt = torch.complex128 if c["precision"] == "fp64" else torch.float32 if real else torch.complex64
    nk, nocc = c["nk"], c["nocc"]
    eo = -0.5 * _uniform(g, (nk, nocc))
    eu = 0.05 + 1.95 * _uniform(g, (nk, max(u for _, u in _sizes(c))))
    Ms, deltas = [], []
    for nb, nu in _sizes(c):
        kq = torch.randperm(nk, generator=g, device="cuda")
        deltas.append((eu[kq][:, None, :nu] - eo[:, :, None]).reshape(-1).contiguous())
        Ms.append(_projections(g, nk * nocc * nu, nb, dt))
    return Ms, deltas


def _screened_inputs(c, seed):
    """P of every q at every frequency (from 2 N_b transitions that stand for 64 x 6,400) and v."""
    g = _gen(seed)
    nb, nw = c["nb"], c["nw"]
    om = torch.as_tensor(_omega(nw), device="cuda")
    v = _coulomb(nb, "cuda")
    rows = 2 * nb
    Ps = []
    for _ in range(c["nq"]):
        M = _projections(g, rows, nb, torch.float32 if c["real"] else torch.complex64)
        d = 0.05 + 2.45 * _uniform(g, (rows,))
        s = (2.0 / 64.0) * (409600.0 / rows) * 2.0 * d / (d * d + om[:, None] ** 2)
        P = torch.empty((nw, nb, nb), dtype=torch.complex128, device="cuda")
        for j in range(nw):
            A = M * s[j].sqrt().float()[:, None]
            H = (A.T @ A.conj()).to(torch.complex128)
            P[j] = -0.5 * (H + H.mH)
        Ps.append(P)
    return Ps, [v] * c["nq"]


def _sigma_inputs(c, seed):
    g = _gen(seed)
    nst, nbd, nb, nw = c["nstates"], c["nbands"], c["nb"], c["nw"]
    dt = torch.complex128 if c["precision"] == "fp64" else torch.complex64
    om = torch.as_tensor(_omega(nw), device="cuda")
    Ms, ps, es, Ws = [], [], [], []
    for _ in range(c["nq"]):
        Ms.append(_projections(g, nst * nbd, nb, dt, MSIG_SCALE))
        nocc = max(1, nbd // 26)
        e = torch.cat([-0.5 * _uniform(g, (nocc,)), 0.05 + 1.95 * _uniform(g, (nbd - nocc,))])
        ps.append(torch.arange(nst, dtype=torch.int32, device="cuda").repeat_interleave(nbd))
        es.append(e.repeat(nst))
        # W^c: Hermitian, negative, of the size v (eps^-1 - 1), falling off with the frequency
        v = _coulomb(nb, "cuda").sqrt()
        X = _projections(g, nb, nb, torch.complex128)
        H = (X @ X.mH) / nb
        H = v[:, None] * H * v[None, :]
        H = 0.5 * (H + H.mH)
        Ws.append(torch.stack([-H / (1.0 + w * w) for w in om.tolist()]))
    return Ms, ps, es, Ws


def _curves(seed, n, nw):
    """Model self-energy curves: 4 to 24 plasmon-shifted poles each (n curves, state signs)."""
    g = _gen(seed)
    z = 1j * torch.as_tensor(_omega(nw), device="cuda")
    npole = 4 + torch.clamp((_uniform(g, (n,)) * 21).long(), max=20)
    sign = torch.where(_uniform(g, (n,)) < 0.5, -1.0, 1.0).to(torch.float64)
    y = torch.zeros((n, nw), dtype=torch.complex128, device="cuda")
    for k in range(24):
        u = _uniform(g, (4, n))
        sg = torch.where(u[0] < 0.5, -1.0, 1.0).to(torch.float64)
        eps = torch.where(u[0] < 0.5, -0.5 * u[1], 0.05 + 1.95 * u[1])
        e = torch.complex(eps + sg * (0.3 + 1.2 * u[2]), -0.01 * sg)
        r = (0.005 + 0.095 * u[3]) * (k < npole)
        y += r[:, None] / (z[None, :] - e[:, None])
    return y, sign


def _byte_buffer(n):
    return torch.empty(int(n), dtype=torch.uint8, device="cuda")


# ---------------------------------------------------------------- the passes
def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"c": c, "om": _omega(c["nw"]) if "nw" in c else _omega(24)}
    if kind in ("polarization", "chain", "real_pw"):
        st["M"], st["d"] = _polar_inputs(c, seed, kind == "real_pw" or c.get("real", False))
        nbs = [m.shape[1] for m in st["M"]]
        st["pref"] = 2.0 / c["nk"]
        if kind != "chain":
            st["P"] = [torch.empty((c["nw"], nb, nb), dtype=torch.complex128, device="cuda")
                       for nb in nbs]
            st["ws"] = _byte_buffer(gw.polarization_workspace(
                [m.shape[0] for m in st["M"]], nbs, c["nw"], c["precision"]))
        st["v"] = [_coulomb(nb, "cuda") for nb in nbs]
        if kind == "chain":
            nbd = c["nocc"] + c["nunocc"]
            st["Ms"], st["ps"], st["es"], _ = _sigma_inputs(
                {"nstates": nbd, "nbands": nbd, "nb": c["nb"], "nw": c["nw"], "nq": c["nq"],
                 "precision": c["precision"]}, seed + 1)
            st["wq"], st["nsig"] = [1.0 / c["nq"]] * c["nq"], nbd
    elif kind == "screened_w":
        st["P"], st["v"] = _screened_inputs(c, seed)
        st["W"] = [torch.empty_like(p) for p in st["P"]]
        if not c["real"]:
            st["ws"] = _byte_buffer(gw.screened_w_workspace([c["nb"]] * c["nq"], c["nw"]))
    elif kind == "sigma":
        st["Ms"], st["ps"], st["es"], st["W"] = _sigma_inputs(c, seed)
        st["wq"] = [1.0 / c["nq"]] * c["nq"]
        st["ws"] = _byte_buffer(gw.sigma_workspace([m.shape[0] for m in st["Ms"]],
                                                   [c["nb"]] * c["nq"], c["nw"], c["precision"]))
    elif kind == "fit":
        st["y"], st["sign"] = _curves(seed, c["n"], c["nw"])
    else:
        st["y"], _ = _curves(seed, c["batch"], 24)
        st["w"] = gw.mlp_init(seed)
        st["g"] = torch.empty_like(st["w"])
    return st


def run(state):
    s, c = state, state["c"]
    kind = c["kind"]
    if kind == "polarization":
        return gw.polarization(s["M"], s["d"], s["om"], s["pref"], c["precision"], out=s["P"],
                               ws=s["ws"])
    if kind == "real_pw":
        P = gw.polarization(s["M"], s["d"], s["om"], s["pref"], c["precision"], out=s["P"],
                            ws=s["ws"])
        return {"P": P, "W": gw.screened_w(P, s["v"], real=True)}
    if kind == "chain":
        P = gw.polarization(s["M"], s["d"], s["om"], s["pref"], c["precision"])
        W = gw.screened_w(P, s["v"])
        sig = gw.sigma_c(s["wq"], s["Ms"], s["ps"], s["es"], W, s["om"], s["om"], s["nsig"],
                         precision=c["precision"])
        return {"P": P, "W": W, "sigma": sig}
    if kind == "screened_w":
        if c["real"]:
            return gw.screened_w(s["P"], s["v"], out=s["W"], real=True)
        return gw.screened_w(s["P"], s["v"], out=s["W"], ws=s["ws"])
    if kind == "sigma":
        return gw.sigma_c(s["wq"], s["Ms"], s["ps"], s["es"], s["W"], s["om"], s["om"],
                          c["nstates"], precision=c["precision"], ws=s["ws"])
    if kind == "fit":
        return gw.continue_fit(s["y"], s["om"], npole=c["npole"], sign=s["sign"])
    # one Adam step from the same weights every time
    w, m, v = s["w"].clone(), torch.zeros_like(s["w"]), torch.zeros_like(s["w"])
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    gw.mlp_train_step(s["y"], s["om"], w, s["g"], m, v, 1e-3, 1, loss)
    return {"w": w, "grad": s["g"], "m": m, "v": v, "loss": loss}


def work(case):
    """Inputs read once and outputs written once, and the operations of the formulas: Hermitian
    results in half the products (4 N_b (N_b + 1) per transition and frequency, complex), the
    factor, inverse and product of a Hermitian solve, the quadratic forms of the pairs, about
    6,000 per iteration and curve of the fit (100 iterations)."""
    c, kind = case, case["kind"]
    b = f = 0.0
    nw = c.get("nw", 24)
    if kind in ("polarization", "chain", "real_pw"):
        real = kind == "real_pw" or c.get("real", False)
        el = 16 if c["precision"] == "fp64" else 4 if real else 8
        for nb, nu in _sizes(c):
            K = c["nk"] * c["nocc"] * nu
            b += K * (nb * el + 8) + 16.0 * nw * nb * nb
            f += (1.0 if real else 4.0) * K * nb * (nb + 1) * nw
            if kind != "polarization":
                b += 16.0 * nw * nb * nb
                f += nw * (1.0 if real else 4.0) * nb ** 3
        if kind == "chain":
            n = c["nocc"] + c["nunocc"]
            b += c["nq"] * n * n * (16.0 * c["nb"] + 12) + 16.0 * n * nw
            f += c["nq"] * 8.0 * n * n * nw * c["nb"] ** 2
    elif kind == "screened_w":
        b = 32.0 * c["nq"] * nw * c["nb"] ** 2
        f = (1.0 if c["real"] else 4.0) * c["nq"] * nw * c["nb"] ** 3
    elif kind == "sigma":
        n = c["nstates"] * c["nbands"]
        el = 16 if c["precision"] == "fp64" else 8
        b = c["nq"] * (n * (el * c["nb"] + 12.0) + 16.0 * nw * c["nb"] ** 2) + 16.0 * c["nstates"] * nw
        f = c["nq"] * 8.0 * n * nw * c["nb"] ** 2
    elif kind == "fit":
        b = c["n"] * (16.0 * nw + 8 + 32.0 * c["npole"] + 16)
        f = c["n"] * 6000.0 * 100
    else:
        b = c["batch"] * 24 * 16.0 + 4.0 * 23816 * 8
        f = c["batch"] * 6.0 * (48 * 128 + 128 * 128 + 128 * 8)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- 64-bit values
def _exact_p(M, d, om, pref):
    """-(pref) sum_t 2 Delta / (Delta^2 + w^2) M_tI conj(M_tJ), from the real parts of M."""
    nb = M.shape[1]
    P = torch.zeros((len(om), nb, nb), dtype=torch.complex128, device="cuda")
    for t0 in range(0, M.shape[0], 32768):
        m, dt = M[t0:t0 + 32768], d[t0:t0 + 32768]
        mr = (m.real if m.is_complex() else m).double()
        mi = m.imag.double() if m.is_complex() else None
        for j, w in enumerate(om):
            s = -pref * 2.0 * dt / (dt * dt + w * w)
            ar = (mr * s[:, None]).T
            if mi is None:
                P[j] += ar @ mr
                continue
            ai = (mi * s[:, None]).T
            C = ar @ mi                                   # sum s Mr_I Mi_J
            P[j] += torch.complex(ar @ mr + ai @ mi, C.T - C)
    return P


def _exact_w(P, v):
    s = v.sqrt()
    out = torch.empty_like(P)
    for j in range(P.shape[0]):
        X = s[:, None] * P[j] * s[None, :]
        L = torch.linalg.cholesky(torch.eye(len(s), dtype=X.dtype, device="cuda") - X)
        Y = s[:, None] * torch.cholesky_solve(X, L) * s[None, :]
        out[j] = 0.5 * (Y + Y.mH)
    return out


def _spline(om):
    """Cardinal cubic splines in lambda = w/(1+w): not-a-knot at the first node, the slope of the
    w^-2 tail at the last. Coefficients [piece][power][node] in powers of lambda - la, piece 0 =
    [0, lambda_0] (the first segment extrapolated), and the pieces' left ends la."""
    n, lam = len(om), om / (1.0 + om)
    h = np.diff(lam)
    A, R = np.zeros((n, n)), np.zeros((n, n))
    E = np.eye(n)
    dl = np.diff(E, axis=0) / h[:, None]                  # divided differences of the unit vectors
    # third derivatives of the first two segments agree
    A[0, :3] = [h[1] ** 2, h[1] ** 2 - h[0] ** 2, -h[0] ** 2]
    R[0] = 2.0 * (h[1] ** 2 * dl[0] - h[0] ** 2 * dl[1])
    for i in range(1, n - 1):
        A[i, i - 1:i + 2] = [h[i], 2.0 * (h[i - 1] + h[i]), h[i - 1]]
        R[i] = 3.0 * (h[i] * dl[i - 1] + h[i - 1] * dl[i])
    A[n - 1, n - 1] = 1.0
    R[n - 1, n - 1] = -2.0 * (1.0 + om[-1]) ** 2 / om[-1]
    m = np.linalg.solve(A, R)
    S = np.zeros((n, 4, n))
    for g in range(n - 1):
        S[g + 1] = [E[g], m[g], (3.0 * dl[g] - 2.0 * m[g] - m[g + 1]) / h[g],
                    (m[g] + m[g + 1] - 2.0 * dl[g]) / h[g] ** 2]
    x, C = -lam[0], S[1]
    S[0] = [C[0] + x * (C[1] + x * (C[2] + x * C[3])), C[1] + x * (2 * C[2] + 3 * x * C[3]),
            C[2] + 3 * x * C[3], C[3]]
    return S, np.concatenate([[0.0], lam[:-1]])


def _exact_convolution(om, energies):
    """T[e][i][j]: the integral over all w' of the interpolant of node values c_j against
    1/(i (w_i + w') - e). With x = w_i + w' = |e| sinh t the kernel is (-i tanh t - sgn(e) sech t)
    dt, smooth in t, so Gauss-Legendre panels in t converge for any e."""
    S, la = _spline(om)
    n = len(om)
    S_t, la_t = torch.as_tensor(S, device="cuda"), torch.as_tensor(la, device="cuda")
    wN = float(om[-1])
    tail = [wN * 2.0 ** k for k in range(8)]
    ends = np.concatenate([[0.0], om, tail[1:]])          # n spline pieces, then 7 tail pieces
    nsub, (gx, gw_) = 16, np.polynomial.legendre.leggauss(16)
    gx, gw_ = torch.as_tensor(gx, device="cuda"), torch.as_tensor(gw_, device="cuda")
    frac = torch.linspace(0, 1, nsub + 1, dtype=torch.float64, device="cuda")
    w = torch.as_tensor(om, device="cuda")
    outs = []
    for e in energies.split(32):
        ae, sg = e.abs()[:, None], torch.sign(e)[:, None]
        T = torch.zeros((len(e), n, n), dtype=torch.complex128, device="cuda")
        for p in range(len(ends) - 1):
            for side in (1.0, -1.0):
                lo, hi = (ends[p], ends[p + 1]) if side > 0 else (-ends[p + 1], -ends[p])
                t0 = torch.asinh((w[None] + lo) / ae)
                t1 = torch.asinh((w[None] + hi) / ae)
                a = t0[..., None] + (t1 - t0)[..., None] * frac        # panel ends
                half = 0.5 * (a[..., 1:] - a[..., :-1])
                t = (0.5 * (a[..., 1:] + a[..., :-1])[..., None] + half[..., None] * gx).flatten(2)
                wt = (half[..., None] * gw_).flatten(2)
                wp = (ae[..., None] * torch.sinh(t) - w[None, :, None]).mul_(side).clamp_(ends[p], ends[p + 1])
                ker = torch.complex(-sg[..., None] / torch.cosh(t), -torch.tanh(t)) * wt
                if p < n:
                    dlam = wp / (1.0 + wp) - la_t[p]
                    f = torch.ones_like(dlam)
                    for k in range(4):
                        T += (ker * f).sum(-1)[..., None] * S_t[p, k]
                        f = f * dlam
                else:
                    T[..., n - 1] += (ker * (wN / wp) ** 2).sum(-1)
        # beyond the last tail piece: w' = X / u on (0, 1]
        X = ends[-1]
        u, wu = 0.5 * (gx + 1.0), 0.5 * gw_
        z = torch.complex(-e[:, None, None] * u, w[None, :, None] * u)
        g = u / (z + 1j * X) + u / (z - 1j * X)
        T[..., n - 1] += (g * wu).sum(-1) * (wN * wN / X)
        outs.append(T)
    return torch.cat(outs)


def _exact_sigma(wq, Ms, ps, es, Ws, om, nsig):
    out = torch.zeros((nsig, len(om)), dtype=torch.complex128, device="cuda")
    for q in range(len(Ms)):
        M = Ms[q].to(torch.complex128)
        c = torch.stack([((M @ Wj.T) * M.conj()).sum(1).real for Wj in Ws[q]])
        ue, inv = torch.unique(es[q], return_inverse=True)
        T = _exact_convolution(om, ue)
        for p in torch.arange(len(inv), device="cuda").split(2048):
            v = torch.einsum("pij,jp->pi", T[inv[p]], c[:, p].to(torch.complex128))
            out.index_add_(0, ps[q][p].long(), v * (-wq[q] / (2.0 * math.pi)))
    return out


def _exact_train(y, w32, om):
    """Loss, gradient and the first Adam step in float64 (autograd)."""
    w = w32.double().requires_grad_(True)
    sizes, at, W = [(128, 48), (128,), (128, 128), (128,), (8, 128), (8,)], 0, []
    for s in sizes:
        W.append(w[at:at + math.prod(s)].reshape(s))
        at += math.prod(s)
    s = y.abs().amax(1)
    s = torch.where(s > 0, s, torch.ones_like(s))
    x = torch.view_as_real(y / s[:, None]).reshape(len(y), -1)
    hid = torch.nn.functional.silu(x @ W[0].T + W[1])
    hid = torch.nn.functional.silu(hid @ W[2].T + W[3])
    o = (hid @ W[4].T + W[5]).reshape(-1, 2, 4)
    z = 1j * torch.as_tensor(om, device="cuda")
    a, p = torch.complex(o[..., 0], o[..., 1]), torch.complex(o[..., 2], o[..., 3])
    fit = (a[..., None] / (z - p[..., None])).sum(1)
    loss = ((fit - y / s[:, None]).abs() ** 2).sum(1).mean() / 24.0
    (g,) = torch.autograd.grad(loss, w)
    m, v = 0.1 * g, 0.001 * g * g
    w = w.detach() - 1e-3 * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    return {"w": w, "grad": g, "m": m, "v": v, "loss": loss.detach().reshape(1)}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "fit" or work(case)["flops"] > 6e12:       # an iteration's end; too long in FP64
        return None
    om = _omega(c.get("nw", 24))
    if kind == "train":
        return _exact_train(_curves(seed, c["batch"], 24)[0], gw.mlp_init(seed), om)
    if kind == "screened_w":
        Ps, vs = _screened_inputs(c, seed)
        return [_exact_w(P, v) for P, v in zip(Ps, vs)]
    if kind == "sigma":
        Ms, ps, es, Ws = _sigma_inputs(c, seed)
        return _exact_sigma([1.0 / c["nq"]] * c["nq"], Ms, ps, es, Ws, om, c["nstates"])
    Ms, ds = _polar_inputs(c, seed, kind == "real_pw" or c.get("real", False))
    P = [_exact_p(M, d, om, 2.0 / c["nk"]) for M, d in zip(Ms, ds)]
    if kind == "polarization":
        return P
    W = [_exact_w(p, _coulomb(p.shape[1], "cuda")) for p in P]
    if kind == "real_pw":
        return {"P": P, "W": W}
    nbd = c["nocc"] + c["nunocc"]
    Ms, ps, es, _ = _sigma_inputs({"nstates": nbd, "nbands": nbd, "nb": c["nb"], "nw": c["nw"],
                                   "nq": c["nq"], "precision": c["precision"]}, seed + 1)
    return {"P": P, "W": W,
            "sigma": _exact_sigma([1.0 / c["nq"]] * c["nq"], Ms, ps, es, W, om, nbd)}
