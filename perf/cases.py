"""Workloads of the library, from its smallest calls to its largest, for timing and for checks of accuracy.

A case is a dict of plain values; `prepare` builds what a program holds before the call (basis, states, G list,
frequencies, a context), `run` makes one pass through the public entry points and `exact` computes the same outputs in
64-bit torch/numpy arithmetic.  Kinds of work:

* ``solve``    one q through the whole path: pair densities, chi0 (direct sum or spectral route), inverse, loss tables;
* ``chi0``     the Adler-Wiser contraction alone, the matrices returned;
* ``pair``     the pair densities alone, returned;
* ``overlap``  overlap matrices of the Bloch sums on a k grid (states preparation);
* ``batch``    heads of uneven (q, w, G_max) instances over several q;
* ``rate``     momentum binning of the loss tables and the halo rate for a heavy and a light mediator;
* ``train``    training of the surrogate network; ``predict`` its inference.

Mixed-precision results are handed on in 32 bits (what the route computes in), FP64 results in 64.  Frequencies reach
40 eV, inside the range of the transition energies (1.1 to 42 eV): above it the loss of these synthetic states is zero but
for isolated poles of width eta, whose height on a frequency grid is a matter of where the grid points fall.
"""
import math

import numpy as np
import torch

from paper_2603_12326_gb300 import qcx

HARTREE_EV = 27.211386245988
BOHR_ANG = 0.529177210903
A_BOHR = 5.43 / BOHR_ANG
UNIT = 2.0 * math.pi / A_BOHR
LATTICE = 0.5 * A_BOHR * np.array([[0.0, 1.0, 1.0], [1.0, 0.0, 1.0], [1.0, 1.0, 0.0]])
ATOMS = np.array([[0.0, 0.0, 0.0], [0.25 * A_BOHR] * 3])
RECIP = 2.0 * np.pi * np.linalg.inv(LATTICE).T
VOLUME = abs(np.linalg.det(LATTICE))
# shells of |q+G| cutoffs of the uneven instances (squares, in units of (2 pi/a)^2)
RADII2 = (4.0, 8.0, 11.0, 12.0, 16.0, 19.0, 20.0, 24.0, 27.0, 32.0, 35.0, 36.0, 40.0, 43.0, 44.0, 48.0)


# ------------------------------------------------------------------------------------------------ the cases
def _physical(name, kind, n_k, shells, nv, nc, ng, nw, wmax=40.0, eta=0.1, prec="mixed", hi=100.0, route="direct",
              nq=1):
    return {"name": name, "kind": kind, "n_k": n_k, "shells": shells, "nv": nv, "nc": nc, "ng": ng, "nw": nw,
            "wmax": wmax, "eta": eta, "prec": prec, "hi": hi, "route": route, "nq": nq}


def listed():
    return [
        # the smallest whole solve: one q of the small workload (4^3 k, N_b 64, N_G 27, 50 w)
        _physical("solve_small", "solve", 4, 8, 4, 12, 27, 50),
        # the ordinary solve, what a production run repeats per q: mid workload, 8^3 k, N_b 96, N_G 181, 200 w
        _physical("solve_mid", "solve", 8, 12, 4, 32, 181, 200),
        # all-electron basis (exponents to 5000 bohr^-2) and the largest G set, on a 4^3 k grid
        _physical("solve_large", "solve", 4, 18, 14, 64, 531, 100, eta=0.05, hi=5000.0),
        # the same ordinary q by the paper's spectral route (grid step eta/20)
        _physical("solve_mid_spectral", "solve", 8, 12, 4, 32, 181, 200, route="spectral"),
        # the FP64 path at a few frequencies: how a user checks the accuracy of the mixed path
        _physical("solve_mid_fp64", "solve", 8, 12, 4, 32, 181, 8, prec="fp64"),
        # pair densities handed to the caller, ordinary size
        _physical("pair_mid", "pair", 8, 12, 4, 32, 181, 1),
        # chi0 matrices handed to the caller, odd sizes throughout (3^3 k, odd bands, N_G not a closed shell)
        _physical("chi0_ragged", "chi0", 3, 9, 5, 23, 113, 37),
        # overlap matrices of the 8^3 k grid: formed once per q when states are prepared
        _physical("overlap_mid", "overlap", 8, 12, 1, 1, 1, 1, prec="fp64"),
        # 256 uneven (q, w, G_max) instances over 10 q of the small workload
        _physical("batch_uneven", "batch", 4, 8, 4, 12, 339, 256, nq=10),
        # the end of a run: binning of 10 q and the halo rate (host results, launch and latency bound)
        _physical("rate_small", "rate", 4, 8, 4, 12, 27, 50, prec="fp64", nq=10),
        # surrogate network: two epochs over the training set of 100 q x 200 w, and inference on a whole grid of heads
        {"name": "mlp_train", "kind": "train", "n": 16257, "epochs": 2, "batch": 256},
        {"name": "mlp_predict", "kind": "predict", "n": 100000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "chi0", "chi0", "pair", "overlap", "batch", "rate", "train", "predict"])
    if kind == "train":
        return {"kind": kind, "n": _log_int(rng, 300, 16257), "epochs": rng.randint(1, 2), "batch": rng.choice([64, 128, 256])}
    if kind == "predict":
        return {"kind": kind, "n": _log_int(rng, 100, 100000)}
    prec = "mixed"
    if kind in ("rate", "overlap") or (kind in ("solve", "chi0", "pair") and rng.random() < 0.25):
        prec = "fp64"
    route = "spectral" if kind == "solve" and rng.random() < 0.25 else "direct"
    eta = rng.choice([0.05, 0.1, 0.1, 0.2])
    wmax = rng.choice([30.0, 40.0, 40.0])
    if kind == "batch":
        c = _physical("", kind, rng.randint(2, 4), rng.randint(4, 8), rng.randint(2, 5), rng.randint(5, 13), 339,
                      _log_int(rng, 16, 256), wmax, eta, nq=rng.randint(2, 10))
    elif kind == "rate":
        c = _physical("", kind, rng.randint(2, 4), rng.randint(4, 8), rng.randint(2, 4), rng.randint(5, 12),
                      _log_int(rng, 9, 27), rng.randint(20, 50), wmax, eta, prec, nq=rng.randint(4, 10))
    elif kind == "overlap":
        c = _physical("", kind, rng.randint(2, 8), rng.randint(4, 12), 1, 1, 1, 1, prec=prec)
    else:
        while True:
            n_k, shells, nv, nc = rng.randint(2, 8), rng.randint(4, 14), rng.randint(2, 9), rng.randint(5, 40)
            ng = _log_int(rng, 9, 339)
            nw = _log_int(rng, 4, 40 if kind == "chi0" else 200) if kind != "pair" else 1
            if prec == "fp64":
                nw = min(nw, 8 if route == "direct" else 20)
            nt = n_k ** 3 * nv * nc
            most = 65536 * 181 ** 2 * (4 if prec == "fp64" else 100)
            span = 41.0 / (eta / (10 if prec == "fp64" else 20))   # points of the spectral grid
            if nt * ng * ng * nw <= most and nt * ng <= 65536 * 181 and \
                    (route == "direct" or span * ng * ng <= (2e7 if prec == "fp64" else 2.7e8)):
                break
        c = _physical("", kind, n_k, shells, nv, nc, ng, nw, wmax, eta, prec, 100.0, route)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------ inputs
def _g_sorted(nmax):
    r = np.arange(-nmax, nmax + 1)
    n = np.stack(np.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)
    g = n @ RECIP
    g2 = np.round(np.einsum("ij,ij->i", g, g), 10)
    return n[np.lexsort((n[:, 2], n[:, 1], n[:, 0], g2))].astype(np.int32)


def _g_ball(q, gmax):
    n = _g_sorted(10)
    k = n @ RECIP + q
    return n[np.einsum("ij,ij->i", k, k) < gmax * gmax]


def _inputs(c, seed):
    """Everything that does not need the overlap of the basis; small arrays, made on the host."""
    rng = np.random.default_rng([26031, seed])
    x = {}
    at, l, ex = [], [], []
    for a in range(2):
        for e in np.sort(np.exp(rng.uniform(np.log(0.1), np.log(c["hi"]), c["shells"]))):
            at += [a, a]
            l += [0, 1]
            ex += [e, e]
    x["shell_atom"], x["shell_l"], x["shell_exp"] = np.array(at, np.int32), np.array(l, np.int32), np.array(ex)
    f = np.array([(i, j, k) for i in range(c["n_k"]) for j in range(c["n_k"]) for k in range(c["n_k"])], float) / c["n_k"]
    x["kpts"] = f @ RECIP
    x["G"] = _g_sorted(8)[:c["ng"]].copy()
    q = []
    while len(q) < c["nq"]:
        d = rng.standard_normal(3)
        v = d / np.linalg.norm(d) * rng.uniform(0.0, 2.0 if c["kind"] == "batch" else 4.0) * UNIT
        if np.min(np.linalg.norm(v + x["G"] @ RECIP, axis=1)) >= 0.1 * UNIT:
            q.append(v)
    x["q"] = np.array(q)
    nk = len(x["kpts"])
    x["Ek"] = np.sort(rng.uniform(-12.0, 0.0, (nk, c["nv"])), axis=-1) / HARTREE_EV
    x["Ekq"] = np.sort(rng.uniform(1.1, 30.0, (c["nq"], nk, c["nc"])), axis=-1) / HARTREE_EV
    x["w"] = np.linspace(0.0, c["wmax"], c["nw"] + 1)[1:] / HARTREE_EV if c["nw"] < 8 else \
        np.linspace(0.0, c["wmax"], c["nw"]) / HARTREE_EV
    x["eta"] = c["eta"] / HARTREE_EV
    if c["kind"] == "batch":
        iq, gm = [], []
        while len(iq) < c["nw"]:
            j, r = int(rng.integers(0, c["nq"])), math.sqrt(RADII2[int(rng.integers(0, len(RADII2)))]) * UNIT
            if np.linalg.norm(x["q"][j]) < r and 15 <= len(_g_ball(x["q"][j], r)) <= 339:
                iq.append(j)
                gm.append(r)
        grid = np.linspace(0.0, c["wmax"], 50)[1:] / HARTREE_EV
        x["inst"] = np.array(iq, np.int32), grid[rng.integers(0, len(grid), len(iq))], np.array(gm)
    return x


def _draws(c, seed):
    """Raw complex-normal coefficient draws at k and, per q, at k+q (device)."""
    g = torch.Generator("cuda").manual_seed(7919 * seed + 13)
    nk, nb = c["n_k"] ** 3, 8 * c["shells"]
    yield torch.randn(nk, nb, c["nv"], dtype=torch.complex128, device="cuda", generator=g)
    for _ in range(c["nq"]):
        yield torch.randn(nk, nb, c["nc"], dtype=torch.complex128, device="cuda", generator=g)


def _orthonormal(S, Z):
    """C with C^H S C = 1 spanning the columns of Z."""
    R = torch.linalg.cholesky(Z.mH @ (S @ Z))
    return torch.linalg.solve_triangular(R, Z.mH, upper=False).mH.resolve_conj().contiguous()


def _states(x, c, seed, overlap):
    zs = _draws(c, seed)
    Ck = _orthonormal(overlap(x["kpts"]), next(zs))
    return Ck, torch.stack([_orthonormal(overlap(x["kpts"] + x["q"][i]), z) for i, z in enumerate(zs)])


def _network(c, seed):
    rng = np.random.default_rng([26032, seed])
    parts = []
    for i, o in ((6, 128), (128, 128), (128, 128), (128, 2)):
        parts += [rng.standard_normal(o * i) / math.sqrt(i), np.zeros(o)]
    n = c["n"]
    d = rng.standard_normal((n, 3))
    X = np.empty((n, 6), np.float32)
    X[:, 0], X[:, 4] = rng.uniform(0.0, 1.0, n), rng.uniform(0.0, 1.0, n)
    X[:, 1:4] = d / np.linalg.norm(d, axis=1)[:, None]
    X[:, 5] = np.log(10.0) * rng.uniform(-4.0, 0.5, n) / 10.0
    y = (-0.5 * np.exp(-X[:, 0]) * (1.0 + 0.3 * np.sin(6.0 * X[:, 4])) + 0.2 * rng.standard_normal(n)).astype(np.float32)
    return np.concatenate(parts).astype(np.float32), X, y


class _State:
    pass


def prepare(case, seed):
    c, s = case, _State()
    s.case = c
    s.stream = torch.cuda.Stream()
    s.ctx = qcx.Context(torch.cuda.current_device(), stream=s.stream.cuda_stream)
    if c["kind"] in ("train", "predict"):
        s.theta, X, y = _network(c, seed)
        s.X, s.y = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
        if c["kind"] == "train":
            s.opts = qcx.mlp_opts(epochs=c["epochs"], batch=c["batch"], seed=seed + 1)
        else:
            s.ctx.mlp_set_params(s.theta)
            s.mu, s.lv = (torch.empty(c["n"], dtype=torch.float32, device="cuda") for _ in range(2))
        torch.cuda.synchronize()
        return s
    x = _inputs(c, seed)
    s.prec = qcx.QCX_FP64 if c["prec"] == "fp64" else qcx.QCX_MIXED
    s.G, s.w, s.eta, s.kpts = x["G"], x["w"], x["eta"], x["kpts"]
    s.ctx.set_basis(LATTICE, ATOMS, x["shell_atom"], x["shell_l"], x["shell_exp"])
    nk, nb = len(x["kpts"]), 8 * c["shells"]
    nt, ng, nw = nk * c["nv"] * c["nc"], c["ng"], c["nw"]

    def empty(*shape, dtype=torch.float64):
        return torch.empty(shape, dtype=dtype, device="cuda")

    def overlap(kpts):
        S = s.ctx.overlap(kpts, out=empty(nk, nb, nb, dtype=torch.complex128))
        s.ctx.sync()
        return S

    if c["kind"] == "overlap":
        s.out = empty(nk, nb, nb, dtype=torch.complex128)
        torch.cuda.synchronize()
        return s
    Ck, Ckq = _states(x, c, seed, overlap)
    torch.cuda.synchronize()
    s.ctx.set_states(x["kpts"], Ck, x["Ek"], x["q"], Ckq, x["Ekq"])
    s.ctx.sync()
    if c["kind"] == "solve":
        s.lfe, s.nolfe = empty(nw, ng), empty(nw, ng)
    elif c["kind"] == "pair":
        s.out = empty(nt, ng, dtype=torch.complex128)
    elif c["kind"] == "chi0":
        s.ctx.pair_density(0, s.G, s.prec)
        s.out = empty(nw, ng, ng, dtype=torch.complex128)
    elif c["kind"] == "batch":
        s.inst = x["inst"]
        s.lfe, s.nolfe = empty(nw), empty(nw)
    elif c["kind"] == "rate":
        for iq in range(c["nq"]):
            s.ctx.pair_density(iq, s.G, s.prec)
            s.ctx.chi0(iq, s.w, s.eta, s.prec)
            s.ctx.invert_eps(iq, s.prec, want=False)
    s.ctx.sync()
    return s


# ------------------------------------------------------------------------------------------------ one pass
EDGES = np.linspace(0.0, 12.0, 121)          # |q+G| bins of the rate, bohr^-1


def _kept(s, *tensors):
    """Results in the precision of the route that computed them."""
    return [t if s.prec == qcx.QCX_FP64 else t.to(torch.complex64 if t.is_complex() else torch.float32) for t in tensors]


def run(state):
    s, c, ctx = state, state.case, state.ctx
    if c["kind"] == "train":
        ctx.mlp_set_params(s.theta)
        curve = ctx.mlp_train(s.X, s.y, s.opts)
        return [ctx.mlp_get_params()[0], curve]
    if c["kind"] == "predict":
        return list(ctx.mlp_predict(s.X, out_mu=s.mu, out_logvar=s.lv))
    if c["kind"] == "rate":
        iqs, nw = list(range(c["nq"])), c["nw"]
        L, count = ctx.bin_loss(iqs, 0, EDGES, nw)
        L2, _ = ctx.bin_loss(iqs, 1, EDGES, nw)
        nz = count > 0
        qb = 0.5 * (EDGES[1:] + EDGES[:-1])[nz]
        heavy = ctx.rate(qb, s.w, L[nz], qcx.halo_params(), nQ=10)
        light = ctx.rate(qb, s.w, L[nz], qcx.halo_params(m_med_eV=0.0), nQ=10)
        return [L, count, L2, *heavy, *light]
    # the library works on the context's own stream
    s.stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s.stream):
        if c["kind"] == "overlap":
            out = [ctx.overlap(s.kpts, out=s.out)]
        elif c["kind"] == "pair":
            out = _kept(s, ctx.pair_density(0, s.G, s.prec, out=s.out))
        elif c["kind"] == "chi0":
            out = _kept(s, ctx.chi0(0, s.w, s.eta, s.prec, out=s.out))
        elif c["kind"] == "batch":
            ctx.solve_batch(*s.inst, s.eta, s.prec, out_lfe=s.lfe, out_nolfe=s.nolfe, want_ng=False)
            out = _kept(s, s.lfe, s.nolfe)
        else:
            ctx.pair_density(0, s.G, s.prec)
            if c["route"] == "spectral":
                step = s.eta / (10 if c["prec"] == "fp64" else 20)
                ctx.chi0_spectral(0, s.w, s.eta, *_grid(ctx, step), s.prec)
            else:
                ctx.chi0(0, s.w, s.eta, s.prec)
            # a check of accuracy looks at the dielectric values too
            eps = ctx.invert_eps(0, s.prec, want=c["prec"] == "fp64")
            ctx.loss_function(0, s.prec, out_lfe=s.lfe, out_nolfe=s.nolfe)
            out = _kept(s, s.lfe, s.nolfe) + ([] if eps is None else list(eps[:2]))
    torch.cuda.current_stream().wait_stream(s.stream)
    return out


def _grid(ctx, step):
    E0, nbin = ctx.spectral_grid(0, step)
    return E0, step, nbin


# ------------------------------------------------------------------------------------------------ work
def _pair_flops(nk, nb, nv, nc, ng):
    return 8.0 * nk * ng * (nb * nb * nv + nb * nv * nc)


def work(case):
    """Each input read and each output written once; the operations of the formulas, with the outer product of each
    transition formed once and one multiply-add per frequency, matrix element and energy resolved at eta/2 (or transition,
    where there are fewer)."""
    c = case
    if c["kind"] in ("train", "predict"):
        per = 2.0 * 33792 * c["n"]
        if c["kind"] == "train":
            return {"bytes": 28.0 * c["n"] * c["epochs"] + 8.0 * 34178, "flops": 3.0 * per * c["epochs"]}
        return {"bytes": 32.0 * c["n"], "flops": per}
    nk, nb = c["n_k"] ** 3, 8 * c["shells"]
    nv, nc, ng, nw = c["nv"], c["nc"], c["ng"], c["nw"]
    nt = nk * nv * nc
    real = 8.0 if c["prec"] == "fp64" else 4.0
    if c["kind"] == "overlap":
        return {"bytes": 16.0 * nk * nb * nb, "flops": 8.0 * nk * nb * nb}
    if c["kind"] == "rate":
        return {"bytes": 8.0 * (2 * c["nq"] * nw * ng + 3 * 120 * nw), "flops": 2.0 * c["nq"] * 2 * nw * ng}
    coef = 2.0 * real * nk * nb * (nv + nc)
    energies = min(nt, 41.0 / (0.5 * c["eta"]))
    chi = 8.0 * ng * ng * (nt + nw * energies)
    if c["kind"] == "pair":
        return {"bytes": coef + 2.0 * real * nt * ng, "flops": _pair_flops(nk, nb, nv, nc, ng)}
    if c["kind"] == "chi0":
        return {"bytes": 2.0 * real * (nt * ng + nw * ng * ng), "flops": chi}
    if c["kind"] == "batch":
        n = float(nw) * 120.0 ** 2            # about the mean square N_G of the instances
        return {"bytes": c["nq"] * coef, "flops": c["nq"] * _pair_flops(nk, nb, nv, nc, ng) + 8.0 * nt * n}
    return {"bytes": coef + 2.0 * real * nw * ng,
            "flops": _pair_flops(nk, nb, nv, nc, ng) + chi + 8.0 * nw * float(ng) ** 3}


# ------------------------------------------------------------------------------------------------ 64-bit values
def _blocks(x, kpts, kappa):
    """Yields (a, b, B[k][G][4][4]) per pair of (s, p_x, p_y, p_z) shell groups: sum_L e^{ik.L} times the Fourier
    integral at kappa of the product of the two Gaussian shells (Gaussian product theorem, every L whose product
    prefactor is at least e^-46)."""
    dev = "cuda"
    at, ex = x["shell_atom"][::2], x["shell_exp"][::2]
    kap = torch.from_numpy(np.ascontiguousarray(kappa)).to(dev)
    kp = torch.from_numpy(np.ascontiguousarray(kpts)).to(dev)
    k2 = (kap * kap).sum(1)
    n = np.stack(np.meshgrid(*[np.arange(-9, 10)] * 3, indexing="ij"), -1).reshape(-1, 3)
    allL = n @ LATTICE
    for a in range(len(ex)):
        for b in range(len(ex)):
            ea, eb, A = ex[a], ex[b], ATOMS[at[a]]
            B = ATOMS[at[b]] + allL
            d2 = np.sum((A - B) ** 2, axis=1)
            keep = d2 * ea * eb / (ea + eb) <= 46.0
            if not keep.any():
                continue
            p = ea + eb
            Bc, Lk = torch.from_numpy(B[keep]).to(dev), torch.from_numpy(allL[keep]).to(dev)
            Ac = torch.from_numpy(A).to(dev)
            P = (ea * Ac + eb * Bc) / p
            K = torch.from_numpy(np.exp(-d2[keep] * ea * eb / p)).to(dev)
            base = (K[:, None] * torch.exp(-k2 / (4.0 * p))) * torch.exp(1j * (P @ kap.T))     # [L][G]
            base = base * ((math.pi / p) ** 1.5 * (2.0 * ea / math.pi) ** 0.75 * (2.0 * eb / math.pi) ** 0.75)
            PA, PB, t = P - Ac, P - Bc, 1j * kap / (2.0 * p)
            e10 = PA[:, None, :] + t                                                            # [L][G][3]
            e01 = PB[:, None, :] + t
            e11 = (PA * PB)[:, None, :] + (PA + PB)[:, None, :] * t + 1.0 / (2.0 * p) - kap * kap / (4.0 * p * p)
            T = torch.empty(*base.shape, 4, 4, dtype=torch.complex128, device=dev)
            na, nb_ = 2.0 * math.sqrt(ea), 2.0 * math.sqrt(eb)
            T[..., 0, 0] = base
            for i in range(3):
                T[..., 1 + i, 0] = base * e10[..., i] * na
                T[..., 0, 1 + i] = base * e01[..., i] * nb_
                for j in range(3):
                    T[..., 1 + i, 1 + j] = base * (e11[..., i] if i == j else e10[..., i] * e01[..., j]) * (na * nb_)
            ph = torch.exp(1j * (kp @ Lk.T))
            yield a, b, (ph @ T.reshape(len(Lk), -1)).reshape(len(kp), len(kap), 4, 4)


def _exact_overlap(x, kpts):
    nb = 2 * len(x["shell_exp"])
    S = torch.zeros(len(kpts), nb, nb, dtype=torch.complex128, device="cuda")
    for a, b, B in _blocks(x, kpts, np.zeros((1, 3))):
        S[:, 4 * a:4 * a + 4, 4 * b:4 * b + 4] = B[:, 0]
    return S


def _exact_rho(x, Ck, Ckq, q, G):
    """rho[t][G], t = (k, v, c)."""
    nk, nb, nv = Ck.shape
    ng, nc = len(G), Ckq.shape[2]
    Y = torch.zeros(nk, nb, ng, nv, dtype=torch.complex128, device="cuda")
    for a, b, B in _blocks(x, x["kpts"], q + G @ RECIP):
        y = B.reshape(nk, ng * 4, 4) @ Ck[:, 4 * b:4 * b + 4]
        Y[:, 4 * a:4 * a + 4] += y.reshape(nk, ng, 4, nv).permute(0, 2, 1, 3)
    r = (Ckq.mH @ Y.reshape(nk, nb, ng * nv)).reshape(nk, nc, ng, nv)
    return r.permute(0, 3, 1, 2).reshape(nk * nv * nc, ng).contiguous()


def _exact_weights(x, iq, w, step=None):
    """W[w][t] of the direct sum, or with hat weights on the energy grid of the given step."""
    dE = torch.from_numpy((x["Ekq"][iq][:, None, :] - x["Ek"][:, :, None]).reshape(-1)).cuda()
    w, z = torch.from_numpy(np.asarray(w)).cuda()[:, None], 1j * x["eta"]

    def kernel(E):
        return 1.0 / (w - E + z) - 1.0 / (w + E + z)

    if step is None:
        return kernel(dE)
    E0 = step * math.floor(float(dE.min()) / step) - step
    u = (dE - E0) / step
    b = torch.floor(u)
    return (1.0 - (u - b)) * kernel(E0 + step * b) + (u - b) * kernel(E0 + step * (b + 1.0))


def _exact_chi0(rho, W, nk):
    return torch.stack([(2.0 / (nk * VOLUME)) * ((rho.mH * Wi) @ rho) for Wi in W])


def _exact_losses(chi, q, G):
    vs = torch.from_numpy(math.sqrt(4.0 * math.pi) / np.linalg.norm(q + G @ RECIP, axis=1)).cuda()
    eps = torch.eye(len(G), dtype=torch.complex128, device="cuda") - vs[:, None] * chi * vs
    inv, diag = torch.linalg.inv(eps).diagonal(dim1=1, dim2=2), eps.diagonal(dim1=1, dim2=2)
    return [-inv.imag, (-1.0 / diag).imag, inv, diag]


def _exact_states(x, c, seed):
    return _states(x, c, seed, lambda kpts: _exact_overlap(x, kpts))


def _exact_rate(q_bohr, w_ha, L, light):
    """dR/dw and recoil spectrum of the truncated-Maxwellian halo (natural units, then events/(kg yr))."""
    alpha, me, hbarc, c = 1.0 / 137.035999084, 510998.95, 1.973269804e-5, 299792.458
    kg, m = 5.609588603804452e35, 1e9
    v0, vesc, vE = 238.0 / c, 544.0 / c, 250.2 / c
    mu = m * me / (m + me)
    pref = 0.3e9 / m * hbarc ** 3 / (2.329 * kg * 1e-3 * hbarc ** 3) * 1e-39 / hbarc ** 2 / (8 * math.pi ** 2 * alpha * mu ** 2)
    y, z = vE / v0, vesc / v0
    norm = 1.0 / (2.0 * (math.erf(z) - 2.0 / math.sqrt(math.pi) * z * math.exp(-z * z)) * v0 * y)

    def eta(v):
        u = v / v0
        if u >= z + y:
            return 0.0
        if u < z - y:
            return norm * (math.erf(u + y) - math.erf(u - y) - 4.0 / math.sqrt(math.pi) * y * math.exp(-z * z))
        return norm * (math.erf(z) - math.erf(u - y) - 2.0 / math.sqrt(math.pi) * (z + y - u) * math.exp(-z * z))

    q, w = q_bohr * alpha * me, w_ha * HARTREE_EV
    F2 = (alpha * me / q) ** 4 if light else np.ones_like(q)
    g = np.array([[qi ** 3 * f * eta(qi / (2 * m) + wj / qi) for wj in w] for qi, f in zip(q, F2)]) * L
    dR = pref * np.sum(0.5 * (g[1:] + g[:-1]) * np.diff(q)[:, None], axis=0) * kg * (365.25 * 86400.0 / 6.582119569e-16)
    step = np.where(w < 1.1, -1, np.floor((w - 1.1) / 3.75)).astype(int)
    return dR, np.array([np.sum(dR[step == k]) * (w[1] - w[0]) for k in range(10)])


def _exact_train(case, seed):
    theta, X, y = _network(case, seed)
    X, y = torch.from_numpy(X).double(), torch.from_numpy(y).double()
    sizes, sel = ((6, 128), (128, 128), (128, 128), (128, 2)), []
    for i, o in sizes:
        sel += [torch.ones(o * i, dtype=torch.bool), torch.zeros(o, dtype=torch.bool)]
    weight, theta = torch.cat(sel), torch.from_numpy(theta).double()

    def nll(p, X, y):
        at, a = 0, X
        for n, (i, o) in enumerate(sizes):
            a = a @ p[at:at + o * i].reshape(o, i).T + p[at + o * i:at + o * i + o]
            a = torch.nn.functional.silu(a) if n < 3 else a
            at += o * i + o
        return a, (0.5 * (a[:, 1] + (y - a[:, 0]) ** 2 * torch.exp(-a[:, 1]))) if y is not None else None

    def rounded(t):                          # the kernels compute with BF16 weights and 32-bit biases
        return torch.where(weight, t.float().bfloat16().double(), t)

    if case["kind"] == "predict":
        a, _ = nll(rounded(theta), X, None)
        return [a[:, 0], a[:, 1]]
    n, mask, s = case["n"], (1 << 64) - 1, seed + 1
    m, v, t, curve = torch.zeros_like(theta), torch.zeros_like(theta), 0, []
    for _ in range(case["epochs"]):
        order = list(range(n))
        for i in range(n - 1, 0, -1):        # Fisher-Yates over splitmix64, the documented shuffle
            s = (s + 0x9E3779B97F4A7C15) & mask
            r = ((s ^ (s >> 30)) * 0xBF58476D1CE4E5B9) & mask
            r = ((r ^ (r >> 27)) * 0x94D049BB133111EB) & mask
            j = (r ^ (r >> 31)) % (i + 1)
            order[i], order[j] = order[j], order[i]
        total = 0.0
        for at in range(0, n, case["batch"]):
            idx = torch.tensor(order[at:at + case["batch"]])
            p = rounded(theta).requires_grad_(True)
            l = nll(p, X[idx], y[idx])[1]
            total += float(l.sum())
            g, = torch.autograd.grad(l.mean(), p)
            t += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            theta = theta - 1e-3 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
        curve.append(total / n)
    return [theta, torch.tensor(curve, dtype=torch.float64)]


def exact(case, seed):
    c = case
    if c["kind"] in ("train", "predict"):
        return _exact_train(c, seed)
    x = _inputs(c, seed)
    if c["kind"] == "overlap":
        return [_exact_overlap(x, x["kpts"])]
    nk, G = len(x["kpts"]), x["G"].astype(np.int64)
    Ck, Ckq = _exact_states(x, c, seed)
    if c["kind"] == "batch":
        inst_q, inst_w, inst_gmax = x["inst"]
        out = torch.empty(2, len(inst_q), dtype=torch.float64)
        for iq in range(c["nq"]):
            mine = np.nonzero(inst_q == iq)[0]
            if not len(mine):
                continue
            Gu = _g_ball(x["q"][iq], inst_gmax[mine].max())
            size = np.linalg.norm(x["q"][iq] + Gu @ RECIP, axis=1)
            rho, W = _exact_rho(x, Ck, Ckq[iq], x["q"][iq], Gu), _exact_weights(x, iq, inst_w[mine])
            for n, i in enumerate(mine):
                cols = np.nonzero(size < inst_gmax[i])[0]
                head = int(np.nonzero((Gu[cols] == 0).all(axis=1))[0][0])
                pick = torch.from_numpy(cols).cuda()
                L = _exact_losses(_exact_chi0(rho[:, pick], W[n:n + 1], nk), x["q"][iq], Gu[cols])
                out[0, i], out[1, i] = L[0][0, head].cpu(), L[1][0, head].cpu()
        return [out[0], out[1]]
    if c["kind"] == "rate":
        L, size = [], []
        for iq in range(c["nq"]):
            rho = _exact_rho(x, Ck, Ckq[iq], x["q"][iq], G)
            L.append(torch.stack(_exact_losses(_exact_chi0(rho, _exact_weights(x, iq, x["w"]), nk), x["q"][iq], G)[:2]))
            size.append(np.linalg.norm(x["q"][iq] + G @ RECIP, axis=1))
        L, size = torch.cat(L, dim=2).cpu().numpy(), np.concatenate(size)            # [2][nw][all G]
        at = np.searchsorted(EDGES, size, side="right") - 1
        n = len(EDGES) - 1
        count = np.array([np.sum(at == b) for b in range(n)], float)
        binned = [np.array([l[:, at == b].sum(axis=1) / max(1.0, count[b]) for b in range(n)]) for l in L]
        nz = count > 0
        qb = 0.5 * (EDGES[1:] + EDGES[:-1])[nz]
        return [binned[0], count, binned[1], *_exact_rate(qb, x["w"], binned[0][nz], False),
                *_exact_rate(qb, x["w"], binned[0][nz], True)]
    rho = _exact_rho(x, Ck, Ckq[0], x["q"][0], G)
    if c["kind"] == "pair":
        return [rho]
    step = x["eta"] / (10 if c["prec"] == "fp64" else 20) if c["route"] == "spectral" else None
    chi = _exact_chi0(rho, _exact_weights(x, 0, x["w"], step), nk)
    return [chi] if c["kind"] == "chi0" else _exact_losses(chi, x["q"][0], G)[:4 if c["prec"] == "fp64" else 2]
