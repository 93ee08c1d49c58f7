"""The calls by which the library's speed is judged.

Each case is one call of the public API on inputs of the shapes and value
distributions of the paper's workloads (band energies with a gap, Gaussian
fit coefficients of variance 1/N_ov, Coulomb matrices with a log-uniform
spectrum, Gauss-Legendre frequencies mapped to [0, inf)).  Sizes come from the
benchmark's workloads, the serving mix and the tests; ``draw`` spreads them
over the whole range of each kind of call.
"""
import math
import random

import numpy as np
import torch

import paper_2505_06021_gb300 as rpa

DEV = "cuda:0"
C128, F64 = torch.complex128, torch.float64
FP64_RATE = 1.9e12  # algorithmic flop/s of the plain FP64 chi0, for the cost of drawn cases
EXACT_FLOPS = 9e12  # FP64 work of the plain 64-bit restatement, at most


def listed():
    return [
        # the serving mix's most frequent job: a Gamma-only molecule, where latency and launches count
        {"name": "gamma_64", "kind": "energy", "grid": 1, "dual": False, "q0": 0, "n_q": 1, "n_aux": 64, "n_occ": 4,
         "n_virt": 28, "n_w": 16, "prec": "fp64", "mem": "device"},
        # a larger Gamma-only cell (ragged sizes of the uneven instances), real data in split precision
        {"name": "gamma_real_mixed", "kind": "energy", "grid": 1, "dual": False, "q0": 0, "n_q": 1, "n_aux": 733,
         "n_occ": 37, "n_virt": 333, "n_w": 16, "prec": "mixed", "mem": "device"},
        # a small periodic cell on the default (FP64) path, 2 x 2 k-points
        {"name": "periodic_fp64", "kind": "energy", "grid": 2, "dual": False, "q0": 0, "n_q": 4, "n_aux": 150,
         "n_occ": 6, "n_virt": 42, "n_w": 12, "prec": "fp64", "mem": "device"},
        # the 2-D periodic benchmark job: 16 q x 16 k, 20 frequencies
        {"name": "periodic2d_mixed", "kind": "energy", "grid": 4, "dual": False, "q0": 0, "n_q": 16, "n_aux": 512,
         "n_occ": 32, "n_virt": 224, "n_w": 20, "prec": "mixed", "mem": "device"},
        # two q-points (one regular, one near Gamma) of the slab dual-grid benchmark job: one rank's block
        {"name": "slab_block", "kind": "energy", "grid": 6, "dual": True, "q0": 7, "n_q": 2, "n_aux": 768, "n_occ": 32,
         "n_virt": 480, "n_w": 16, "prec": "mixed", "mem": "device"},
        # inputs in pinned host memory, staged by the library (a user's job that does not live on the GPU)
        {"name": "host_staged", "kind": "energy", "grid": 2, "dual": False, "q0": 0, "n_q": 4, "n_aux": 300,
         "n_occ": 20, "n_virt": 130, "n_w": 16, "prec": "mixed", "mem": "host"},
        # the response step alone for one q on the default (FP64) path
        {"name": "chi0_fp64_q", "kind": "chi0", "grid": 3, "dual": False, "q0": 1, "n_q": 2, "n_aux": 320, "n_occ": 16,
         "n_virt": 120, "n_w": 16, "prec": "fp64"},
        # the log-det step alone for one q of the slab job
        {"name": "logdet_q", "kind": "logdet", "cplx": True, "n_aux": 768, "n_w": 16, "noalloc": False},
        # the allocation-free log-det, a ragged size of its range
        {"name": "logdet_noalloc", "kind": "logdet", "cplx": True, "n_aux": 201, "n_w": 12, "noalloc": True},
        # AO -> MO transform of the fit coefficients for one q, 4 x 4 k-points
        {"name": "ao2mo_q", "kind": "ao2mo", "grid": 4, "n_atoms": 2, "nb": 96, "nf": 192, "n_occ": 32, "n_virt": 160},
        # periodic projector on the benchmark's basis size
        {"name": "projector", "kind": "projector", "grid": 4, "n_atoms": 2, "nb": 128, "n_mo": 256},
        # many independent uneven jobs in one call
        {"name": "batch_uneven", "kind": "batch", "n_jobs": 12, "aux_lo": 128, "aux_hi": 640, "occ_hi": 20, "n_w": 16,
         "sizes": 11},
    ]


# ------------------------------------------------------------------ drawing


def _logint(r, lo, hi):
    return int(round(math.exp(r.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["energy", "energy", "energy", "chi0", "logdet", "logdet", "ao2mo", "projector", "batch"])
    while True:
        c = {"kind": kind}
        if kind in ("energy", "chi0"):
            grid = rng.choice([1, 2, 2, 3, 4])
            c.update(grid=grid, dual=False, q0=0, n_aux=_logint(rng, 48, 768), n_occ=_logint(rng, 4, 40),
                     n_w=rng.randint(8, 24), prec=rng.choice(["fp64", "mixed"]))
            c["n_virt"] = c["n_occ"] * rng.randint(4, 12) + rng.randint(0, 3)
            c["n_q"] = 1 if grid == 1 else rng.randint(1, min(grid * grid, 4))
            if kind == "energy":
                c["mem"] = "host" if rng.random() < 0.15 else "device"
        elif kind == "logdet":
            noalloc = rng.random() < 0.4
            c.update(cplx=rng.random() < 0.75, n_aux=_logint(rng, 48, 384 if noalloc else 900),
                     n_w=rng.randint(6, 20), noalloc=noalloc)
        elif kind == "ao2mo":
            c.update(grid=rng.choice([1, 2, 3, 4]), n_atoms=rng.randint(1, 3), nb=_logint(rng, 16, 100))
            c["nf"] = c["nb"] * 2 + rng.randint(-3, 3)
            c["n_occ"] = max(1, c["n_atoms"] * c["nb"] // rng.randint(6, 10))
            c["n_virt"] = c["n_atoms"] * c["nb"] - c["n_occ"] - rng.randint(0, 2)
        elif kind == "projector":
            c.update(grid=rng.choice([1, 2, 3, 4]), n_atoms=rng.randint(1, 3), nb=_logint(rng, 20, 85))
            c["n_mo"] = c["n_atoms"] * c["nb"] - rng.randint(0, 5)
        else:
            c.update(n_jobs=rng.randint(4, 12), aux_lo=64, aux_hi=rng.randint(128, 512), occ_hi=rng.randint(8, 20),
                     n_w=rng.randint(8, 16), sizes=rng.randint(0, 10**6))
        w = work(c)
        fp64 = c.get("prec") == "fp64" or kind in ("ao2mo",)
        if w["flops"] <= (0.7 * FP64_RATE if fp64 else 2e13) and w["bytes"] <= 6e9:
            if c.get("mem") != "host" or w["bytes"] <= 1.5e9:
                return c


# ------------------------------------------------------------------- inputs


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, shape, cplx, var):
    """Gaussian entries of the given variance (complex: split over re and im)."""
    if not cplx:
        return torch.randn(shape, generator=g, device=DEV, dtype=F64).mul_(math.sqrt(var))
    x = torch.randn(tuple(shape) + (2,), generator=g, device=DEV, dtype=F64).mul_(math.sqrt(0.5 * var))
    return torch.view_as_complex(x)


def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device=DEV, dtype=F64) * (hi - lo) + lo


def _haar(g, n, cplx):
    q, r = torch.linalg.qr(_randn(g, (n, n), cplx, 1.0))
    d = torch.diagonal(r)
    return q * (d / d.abs())[None, :]


def _hermitian(q, lam):
    m = (q * lam[None, :].to(q.dtype)) @ q.conj().T
    return (0.5 * (m + m.conj().T)).contiguous()


def _coulomb(g, n, cplx):
    return _hermitian(_haar(g, n, cplx), torch.exp(_uniform(g, n, math.log(0.1), math.log(10.0))))


def _freqs(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return (1.0 + x) / (1.0 - x), w * 2.0 / (1.0 - x) ** 2


def _grid(n, dual):
    """(pair_k, pair_kq, w_q, zeta_k, kpts): an n x n grid with q on the same
    grid, or the dual grid: q on the n/2 x n/2 grid without Gamma plus four
    points near Gamma."""
    k = [(i / n, j / n) for i in range(n) for j in range(n)]
    kpts, pk, pkq, wq = list(k), [], [], []
    m = n // 2 if dual else n
    step = n // m
    for a in range(m):
        for b in range(m):
            if dual and a == b == 0:
                continue
            pk.append(list(range(n * n)))
            pkq.append([((i + a * step) % n) * n + (j + b * step) % n for i in range(n) for j in range(n)])
            wq.append(1.0 / m**2)
    if dual:
        d = 0.1 / m
        for sx, sy in ((-d, -d), (-d, d), (d, -d), (d, d)):
            pk.append(list(range(n * n)))
            pkq.append([len(kpts) + i for i in range(n * n)])
            kpts += [(x + sx, y + sy) for x, y in k]
            wq.append(0.25 / m**2)
    return np.array(pk), np.array(pkq), np.array(wq), 1.0 / n**2, np.array(kpts)


def _bands(g, kpts, n_occ, n_virt):
    occ = torch.sort(_uniform(g, n_occ, -1.0, -0.3)).values
    virt = torch.sort(_uniform(g, n_virt, 0.1, 2.0)).values
    disp = 0.0 if len(kpts) == 1 else 0.05
    shift = torch.from_numpy(disp * 0.5 * np.cos(2 * np.pi * kpts).sum(1)).to(DEV)
    return (occ[None, :] + shift[:, None]).contiguous(), (virt[None, :] + shift[:, None]).contiguous()


def _response_inputs(c, seed):
    g = _gen(seed)
    cplx = c["grid"] > 1
    pk, pkq, wq, zeta, kpts = _grid(c["grid"], c["dual"])
    sel = slice(c["q0"], c["q0"] + c["n_q"])
    pk, pkq, wq = pk[sel], pkq[sel], wq[sel]
    nov, n_k = c["n_occ"] * c["n_virt"], pk.shape[1]
    eo, ev = _bands(g, kpts, c["n_occ"], c["n_virt"])
    om, zw = _freqs(c["n_w"])
    n = pk.size
    C = _randn(g, (n, c["n_aux"], nov), cplx, 1.0 / nov)
    V = [_coulomb(g, c["n_aux"], cplx) for _ in range(len(wq))]
    return dict(cplx=cplx, pk=pk, pkq=pkq, wq=wq, zeta=zeta, eo=eo, ev=ev, om=om, zw=zw, C=C, V=V, n_k=n_k)


def _job(c, d):
    host = c.get("mem") == "host"

    def put(t):
        if not host:
            return t
        h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
        return h.copy_(t)

    C = put(d["C"])
    return rpa.Job(is_complex=d["cplx"], n_aux=c["n_aux"], n_occ=c["n_occ"], n_virt=c["n_virt"], pair_k=d["pk"],
                   pair_kq=d["pkq"], w_q=d["wq"], zeta_k=d["zeta"], omega=d["om"], zeta_w=d["zw"], eps_occ=put(d["eo"]),
                   eps_virt=put(d["ev"]), C=[C[i] for i in range(C.shape[0])], V=[put(v) for v in d["V"]],
                   prec=rpa.PREC_MIXED if c["prec"] == "mixed" else rpa.PREC_FP64,
                   mem=rpa.MEM_HOST if host else rpa.MEM_DEVICE)


def _batch_cases(c):
    """The jobs of a batch: Gamma-only real or 2 x 2 complex, split precision,
    every fourth one on the FP64 path and small."""
    r = random.Random(c["sizes"])
    out = []
    for i in range(c["n_jobs"]):
        fp64 = i % 4 == 3
        n_occ = r.randint(4, c["occ_hi"])
        grid = r.choice([1, 2])
        out.append({"grid": grid, "dual": False, "q0": 0, "n_q": grid * grid,
                    "n_aux": r.randint(c["aux_lo"], min(c["aux_hi"], 160) if fp64 else c["aux_hi"]), "n_occ": n_occ,
                    "n_virt": n_occ * r.randint(4, 10), "n_w": c["n_w"], "prec": "fp64" if fp64 else "mixed"})
    return out


def _chi_inputs(c, seed):
    """V and a negative semidefinite response that falls off with the frequency."""
    g = _gen(seed)
    n = c["n_aux"]
    V = _coulomb(g, n, c["cplx"])
    om, _ = _freqs(c["n_w"])
    chi = torch.empty((c["n_w"], n, n), dtype=C128 if c["cplx"] else F64, device=DEV)
    A = _randn(g, (2 * n, n), c["cplx"], 0.5 / n)
    gap = torch.linspace(0.4, 3.0, 2 * n, dtype=F64, device=DEV)
    for w in range(c["n_w"]):
        d = -4.0 * gap / (gap * gap + float(om[w]) ** 2)
        x = (A.conj().T * d[None, :].to(A.dtype)) @ A
        chi[w] = 0.5 * (x + x.conj().T)
    return V, chi


def _ao_inputs(c, seed):
    g = _gen(seed)
    cplx = c["grid"] > 1
    pk, pkq, wq, zeta, kpts = _grid(c["grid"], False)
    N = c["n_atoms"] * c["nb"]
    nf = c.get("nf", 1)
    n_occ = c.get("n_occ", max(1, c.get("n_mo", 2) // 8))
    n_virt = c.get("n_virt", c.get("n_mo", 2) - n_occ)
    n_mo = c.get("n_mo", n_occ + n_virt)
    nk = len(kpts)
    eo, ev = _bands(g, kpts, n_occ, n_virt)
    S = N * nf
    padf = [_randn(g, (N, S), cplx, c["n_atoms"] / (2.0 * n_occ * n_virt)) for _ in range(nk)]
    mo = [_haar(g, N, cplx)[:, :n_mo].contiguous() for _ in range(nk)]
    ovl = None
    if c["kind"] == "projector":
        ovl = []
        for k in range(nk):
            lam = _uniform(g, N, 0.3, 3.0)
            n_small = (int(seed) + k) % 4
            lam[:n_small] = torch.exp(_uniform(g, n_small, math.log(1e-7), math.log(1e-5)))
            ovl.append(_hermitian(_haar(g, N, cplx), lam))
    n_aux = c["n_atoms"] * nf
    V = [_coulomb(g, n_aux, cplx) for _ in range(len(wq) if c["kind"] == "projector" else 2)]
    return dict(cplx=cplx, pk=pk, pkq=pkq, wq=wq, zeta=zeta, eo=eo, ev=ev, padf=padf, mo=mo, ovl=ovl, V=V, N=N,
                n_aux=n_aux, n_occ=n_occ, n_virt=n_virt, n_mo=n_mo, q=len(wq) - 1)


# ---------------------------------------------------------------- the calls

_CTX = []


def _ctx():
    """The library context that a program opens once and keeps."""
    if not _CTX:
        _CTX.append(rpa.Context(0))
    return _CTX[0]


def prepare(case, seed):
    k = case["kind"]
    s = {"kind": k, "case": case}
    if k in ("energy", "chi0"):
        s["job"] = _job(case, _response_inputs(case, seed))
    elif k == "batch":
        s["jobs"] = [_job(c, _response_inputs(c, seed * 1000 + i)) for i, c in enumerate(_batch_cases(case))]
    elif k == "logdet":
        V, chi = _chi_inputs(case, seed)
        s["V"], s["chi"] = V, chi
        if case["noalloc"]:
            s["out"] = torch.empty((case["n_w"], 2), dtype=F64, device=DEV)
        else:
            om, zw = _freqs(case["n_w"])
            one = torch.ones((1, 1), dtype=F64, device=DEV)
            C = torch.ones((case["n_aux"], 1), dtype=chi.dtype, device=DEV)
            z = np.zeros((1, 1), np.int32)
            s["job"] = rpa.Job(is_complex=case["cplx"], n_aux=case["n_aux"], n_occ=1, n_virt=1, pair_k=z, pair_kq=z,
                               w_q=np.ones(1), zeta_k=1.0, omega=om, zeta_w=zw, eps_occ=-one, eps_virt=one, C=[C],
                               V=[V])
    else:
        d = _ao_inputs(case, seed)
        V = [d["V"][min(i, len(d["V"]) - 1)] for i in range(len(d["wq"]))]
        ao = {"n_bas_atom": [case["nb"]] * case["n_atoms"], "n_fit_atom": [case.get("nf", 1)] * case["n_atoms"],
              "padf": d["padf"], "mo": d["mo"]}
        if k == "projector":
            ao.update(overlap=d["ovl"], eps_d=1e-4)
        om, zw = _freqs(4)
        s["job"] = rpa.Job(is_complex=d["cplx"], n_aux=d["n_aux"], n_occ=d["n_occ"], n_virt=d["n_virt"],
                           pair_k=d["pk"], pair_kq=d["pkq"], w_q=d["wq"], zeta_k=d["zeta"], omega=om, zeta_w=zw,
                           eps_occ=d["eo"], eps_virt=d["ev"], C=None, V=V, ao=ao)
        s["q"] = d["q"]
    _ctx()
    torch.cuda.synchronize()
    return s


def run(state):
    k, ctx = state["kind"], _ctx()
    if k == "energy":
        return ctx.energy(state["job"])
    if k == "batch":
        return ctx.energy_batch(state["jobs"])
    if k == "chi0":
        return ctx.chi0(state["job"], state["job"].n_q - 1)
    if k == "logdet":
        if state["case"]["noalloc"]:
            c = state["case"]
            rpa.logdet_noalloc(c["cplx"], c["n_aux"], c["n_w"], state["V"], state["chi"], state["out"])
            return state["out"]
        return ctx.logdet(state["job"], 0, state["chi"])
    if k == "ao2mo":
        return ctx.ao2mo(state["job"], state["q"])
    out, m, eig = ctx.projector(state["job"])
    return {"mo": out, "removed": m, "eig": eig}


# ------------------------------------------------------------------- work


def _response_work(c, n_q):
    cplx = c["grid"] > 1
    es, f = (16, 4.0) if cplx else (8, 1.0)
    N, nov, n_k = c["n_aux"], c["n_occ"] * c["n_virt"], c["grid"] ** 2
    byt = es * (N * nov * n_k + N * N) * n_q
    return byt, f * N * (N + 1) * nov * n_k * c["n_w"] * n_q


def _logdet_flops(cplx, N, n_w):
    # V = L L^H, the two triangular products, the factorisation: multiply and add per (complex) entry
    return (8.0 if cplx else 2.0) * N**3 * (1.0 / 6 + n_w * (1.0 / 6 + 2.0 / 3))


def work(case):
    k = case["kind"]
    if k in ("energy", "chi0"):
        n_q = 1 if k == "chi0" else case["n_q"]
        byt, fl = _response_work(case, n_q)
        if k == "chi0":
            return {"bytes": byt + (16 if case["grid"] > 1 else 8) * case["n_aux"] ** 2 * case["n_w"], "flops": fl}
        return {"bytes": byt, "flops": fl + n_q * _logdet_flops(case["grid"] > 1, case["n_aux"], case["n_w"])}
    if k == "batch":
        w = [work(dict(c, kind="energy")) for c in _batch_cases(case)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    if k == "logdet":
        return {"bytes": (16 if case["cplx"] else 8) * case["n_aux"] ** 2 * (case["n_w"] + 1),
                "flops": _logdet_flops(case["cplx"], case["n_aux"], case["n_w"])}
    cplx = case["grid"] > 1
    es, f = (16, 8.0) if cplx else (8, 2.0)
    nk, N = case["grid"] ** 2, case["n_atoms"] * case["nb"]
    if k == "ao2mo":
        S, nov = N * case["nf"], case["n_occ"] * case["n_virt"]
        n_mo = case["n_occ"] + case["n_virt"]
        return {"bytes": es * nk * (N * S + N * n_mo + case["n_atoms"] * case["nf"] * nov),
                "flops": f * nk * (S * N * n_mo + 2.0 * S * nov)}
    # eigenvalues of every overlap (reduction to tridiagonal form) and the rank-m projection
    return {"bytes": es * nk * (N * N + 2 * N * case["n_mo"]), "flops": f * nk * (2.0 / 3) * N**3}


# ------------------------------------------- plain restatements in 64 bits


def _eps_of(V, chi):
    """(ln det(1 - Pi), Tr Pi) for Pi = L^H chi L, V = L L^H (the same determinant
    and trace as with V^(1/2))."""
    L = torch.linalg.cholesky(V)
    Y = L.conj().T @ chi @ L
    M = torch.eye(V.shape[0], dtype=V.dtype, device=V.device) - 0.5 * (Y + Y.conj().T)
    ld = 2.0 * torch.log(torch.diagonal(torch.linalg.cholesky(M)).real).sum()
    return float(ld), float(torch.diagonal(Y).real.sum())


def _chi_of(c, d, q, w):
    chi = 0
    for j in range(d["n_k"]):
        D = d["ev"][d["pkq"][q, j]][None, :] - d["eo"][d["pk"][q, j]][:, None]
        wt = (d["zeta"] * (-4.0 * D / (D * D + float(d["om"][w]) ** 2))).reshape(-1)
        C = d["C"][q * d["n_k"] + j]
        chi = chi + (C.conj() * wt[None, :]) @ C.T
    return chi


def _energy_exact(c, seed):
    d = _response_inputs(c, seed)
    n_q, n_w = len(d["wq"]), c["n_w"]
    ld, tr = np.zeros((n_q, n_w)), np.zeros((n_q, n_w))
    for q in range(n_q):
        for w in range(n_w):
            ld[q, w], tr[q, w] = _eps_of(d["V"][q], _chi_of(c, d, q, w))
    eps = ld + tr
    Ec = float((d["wq"][:, None] * d["zw"][None, :] * eps).sum() / (2.0 * math.pi))
    return {"Ec": Ec, "eps": eps, "lndet": ld, "trPi": tr}


def exact(case, seed):
    k = case["kind"]
    if k in ("energy", "chi0", "batch") and 2.0 * work(case)["flops"] > EXACT_FLOPS:
        return None
    if k == "energy":
        return _energy_exact(case, seed)
    if k == "batch":
        return np.array([_energy_exact(c, seed * 1000 + i)["Ec"] for i, c in enumerate(_batch_cases(case))])
    if k == "chi0":
        d = _response_inputs(case, seed)
        return torch.stack([_chi_of(case, d, len(d["wq"]) - 1, w) for w in range(case["n_w"])])
    if k == "logdet":
        V, chi = _chi_inputs(case, seed)
        r = np.array([_eps_of(V, chi[w]) for w in range(case["n_w"])])
        return torch.from_numpy(r).to(DEV) if case["noalloc"] else r
    d = _ao_inputs(case, seed)
    if k == "projector":
        eig, U = zip(*[torch.linalg.eigh(s) for s in d["ovl"]])
        m = max(int((e < 1e-4).sum()) for e in eig)
        out = [c - u[:, :m] @ (u[:, :m].conj().T @ c) for u, c in zip(U, d["mo"])]
        return {"mo": out, "removed": None, "eig": torch.stack(eig).cpu().numpy()}
    q, no, nb, nf = d["q"], d["n_occ"], case["nb"], case["nf"]
    C = torch.empty((d["pk"].shape[1], d["n_aux"], no * d["n_virt"]), dtype=C128 if d["cplx"] else F64, device=DEV)
    for j in range(d["pk"].shape[1]):
        kk, kq = int(d["pk"][q, j]), int(d["pkq"][q, j])
        Ho, Hv = d["padf"][kk].T @ d["mo"][kk][:, :no], d["padf"][kq].T @ d["mo"][kq][:, no:]
        for A in range(case["n_atoms"]):
            b, s = slice(A * nb, (A + 1) * nb), slice(A * nb * nf, (A + 1) * nb * nf)
            x = torch.einsum("mi,mga->gia", d["mo"][kk][b, :no].conj(), Hv[s].reshape(nb, nf, -1))
            x = x + torch.einsum("na,ngi->gia", d["mo"][kq][b, no:], Ho[s].reshape(nb, nf, no).conj())
            C[j, A * nf:(A + 1) * nf] = x.reshape(nf, -1)
    return C
