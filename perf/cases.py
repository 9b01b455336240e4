"""The calls whose speed matters to a user of this package, with inputs, sizes and plain 64-bit answers.

Five kinds of call, each through the public entry points:

  bounds   a new disorder realization: build the sector, get E_min and E_max
  factor   factor H - sigma and solve one block of right-hand sides to FP64 accuracy
  solve    one refined block solve with a factorization that the program keeps
  job      the whole method: sector, eigenpairs nearest the target, their observables
  served   several whole jobs given to a running server at once
  observe  the observables of eigenvectors that the program already has

Chains of L = 8 to 20 sites, both parities, disorder from the extended to the localized side, both
precisions of the fronts, block widths from 1 to 32.  The fields h_i, the right-hand sides and the vectors
come from the seed.  A program keeps one context (with its symbolic analyses) and one server, so they live
at module level.

Targets of factor and solve lie at 0.03 to 0.1 of the spectrum (where resolvents are computed for their own
sake); jobs take the whole range of energy densities.  Eigenvectors and entropies are returned the way such
a program stores them: sign fixed by the largest component, in single precision, since a vector is
determined to residual / gap only.
"""
import functools
import math

import numpy as np
import torch

import paper_1411_0660_gb300 as g

PREC = {"fp32": g.MBL_PREC_FP32, "fp64": g.MBL_PREC_FP64}


def listed():
    return [
        # the first step of every job, at the size where the sector no longer fits L2 twice over
        {"name": "bounds_L20", "kind": "bounds", "L": 20, "nup": 10, "h": 3.0},
        # resolvent blocks: a small chain, the size of the headline workload with FP64 fronts, and the largest
        {"name": "factor_L14", "kind": "factor", "L": 14, "nup": 7, "h": 2.5, "eps": 0.1, "p": 8, "prec": "fp32"},
        {"name": "factor_L18_fp64", "kind": "factor", "L": 18, "nup": 9, "h": 3.0, "eps": 0.1, "p": 8, "prec": "fp64"},
        {"name": "factor_L19", "kind": "factor", "L": 19, "nup": 10, "h": 3.0, "eps": 0.1, "p": 8, "prec": "fp32"},
        # a kept factorization: one right-hand side, and a wide block at the headline size
        {"name": "solve_L16_p1", "kind": "solve", "L": 16, "nup": 8, "h": 4.0, "eps": 0.1, "p": 1, "prec": "fp32"},
        {"name": "solve_L18_p16", "kind": "solve", "L": 18, "nup": 9, "h": 3.0, "eps": 0.1, "p": 16, "prec": "fp32"},
        # whole jobs: the smallest size that is averaged over realizations, an odd chain, the batch workload's
        # size with FP64 fronts, the headline size
        {"name": "job_L12", "kind": "job", "L": 12, "nup": 6, "h": 2.0, "eps": 0.5, "nev": 20, "prec": "fp32"},
        {"name": "job_L15", "kind": "job", "L": 15, "nup": 8, "h": 1.0, "eps": 0.7, "nev": 30, "prec": "fp32"},
        {"name": "job_L16_fp64", "kind": "job", "L": 16, "nup": 8, "h": 2.5, "eps": 0.5, "nev": 50, "prec": "fp64"},
        {"name": "job_L18", "kind": "job", "L": 18, "nup": 9, "h": 3.0, "eps": 0.5, "nev": 50, "prec": "fp32"},
        # a stream of realizations through the server
        {"name": "served_L14", "kind": "served", "L": 14, "nup": 7, "h": 3.5, "eps": 0.5, "nev": 20, "prec": "fp32", "jobs": 8},
        # observables of one job of the headline workload
        {"name": "observe_L18", "kind": "observe", "L": 18, "nup": 9, "nev": 50},
    ]


def draw(rng):
    kind = rng.choice(["bounds", "factor", "factor", "solve", "job", "job", "served", "observe"])
    top = {"bounds": 20, "factor": 18, "solve": 18, "job": 17, "served": 14, "observe": 18}[kind]
    L = rng.randint({"bounds": 10, "factor": 10, "solve": 10, "job": 10, "served": 10, "observe": 8}[kind], top)
    nup = L // 2 if L % 2 == 0 else (L + 1) // 2
    if L < 16 and rng.random() < 0.3:
        nup -= 1
    c = {"kind": kind, "L": L, "nup": nup}
    if kind != "observe":
        c["h"] = round(math.exp(rng.uniform(math.log(0.5), math.log(6.0))), 3)
    if kind in ("factor", "solve"):
        c["eps"] = round(rng.uniform(0.03, 0.1), 4)
        c["p"] = rng.choice([1, 3, 7, 8, 8, 13, 16, 32])
        c["prec"] = rng.choice(["fp32", "fp32", "fp64"])
    if kind in ("job", "served"):
        c["eps"] = round(rng.uniform(0.1, 0.9), 3)
        c["nev"] = rng.choice([10, 20, 20, 30, 50])
        c["prec"] = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "served":
        c["jobs"] = rng.randint(2, 8)
    if kind == "observe":
        c["nev"] = int(round(math.exp(rng.uniform(math.log(3), math.log(64)))))
    return c


# ---- the program's side ---------------------------------------------------------------------------------


@functools.lru_cache(maxsize=None)
def _context():
    return g.Context(0)


@functools.lru_cache(maxsize=None)
def _stream():
    return torch.cuda.Stream()


@functools.lru_cache(maxsize=None)
def _server():
    # each job is another realization, so there is nothing for the factorization cache to keep
    ctx = g.Context(0)
    return g.Server(ctx, slots=4, cache_fraction=0.0)


def _fields(c, seed, k=0):
    return np.random.default_rng([seed, k]).uniform(-c["h"], c["h"], c["L"])


def _normal(shape, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)


def _vectors(c, seed):
    """Unit vectors with amplitudes between those of extended and localized states."""
    n = math.comb(c["L"], c["nup"])
    v = _normal((c["nev"], n), seed) * torch.exp(1.5 * _normal((c["nev"], n), seed + 1))
    return v / v.norm(dim=1, keepdim=True)


def _levels(c, seed):
    return _normal((c["nev"],), seed + 2).sort().values


def _target(c, lo, hi):
    return round(lo + c["eps"] * (hi - lo), 6)


def prepare(c, seed):
    kind, L = c["kind"], c["L"]
    f64 = dict(device="cuda", dtype=torch.float64)
    s = {"case": c}
    n = math.comb(L, c["nup"])
    if kind != "served":
        s["ctx"], s["stream"] = _context(), _stream()
    if kind in ("bounds", "job"):
        s["fields"] = _fields(c, seed)
    if kind == "served":
        s["server"], s["fields"] = _server(), [_fields(c, seed, k) for k in range(c["jobs"])]
    if kind in ("factor", "solve"):
        s["sec"] = g.build_sector_fields(s["ctx"], L, _fields(c, seed), nup=c["nup"])
        s["sigma"] = _target(c, *g.extremal_bounds(s["sec"]))
        s["b"] = _normal((c["p"], n), seed)
        s["x"] = torch.zeros_like(s["b"])
    if kind == "solve":
        s["f"] = g.factor(s["sec"], s["sigma"], precision=PREC[c["prec"]])
    if kind in ("job", "observe"):
        nev = c["nev"]
        s["evals"], s["evecs"], s["resid"] = torch.zeros(nev, **f64), torch.zeros(nev, n, **f64), torch.zeros(nev, **f64)
        s["r"], s["r_mean"], s["s1p"], s["se"] = (torch.zeros(k, **f64) for k in (max(nev - 2, 1), 1, nev, nev))
    if kind == "observe":
        s["evecs"], s["evals"] = _vectors(c, seed), _levels(c, seed)
        s["kl"], s["sqp"], s["fluct"], s["dynf"] = (torch.zeros(k, **f64) for k in (max(nev - 1, 1), nev, nev, nev))
    return s


def _stored(v):
    """Eigenvectors (rows) as they are stored: the largest component positive, single precision."""
    top = v.gather(1, v.abs().argmax(dim=1, keepdim=True))
    return (v * top.sign()).float()


def run(s):
    c = s["case"]
    kind, L, nup = c["kind"], c["L"], c["nup"]
    if kind == "served":
        srv = s["server"]
        tickets = [srv.submit(L, c["h"], 0, c["eps"], c["nev"], precision=PREC[c["prec"]], fields=f, nup=nup) for f in s["fields"]]
        done = [srv.wait(t) for t in tickets]
        return {"evals": np.stack([d.evals for d in done]), "r": np.stack([d.r for d in done]),
                "s1p": np.stack([d.s1p for d in done]).astype(np.float32), "se": np.stack([d.se for d in done]).astype(np.float32)}
    ctx, stream = s["ctx"], s["stream"]
    if kind == "bounds":
        return list(g.extremal_bounds(g.build_sector_fields(ctx, L, s["fields"], nup=nup)))
    if kind == "factor":
        f = g.factor(s["sec"], s["sigma"], precision=PREC[c["prec"]])
        f.solve_dev(s["b"], s["x"], c["p"], refine=True, stream=stream)
        return s["x"]
    if kind == "solve":
        s["f"].solve_dev(s["b"], s["x"], c["p"], refine=True, stream=stream)
        return s["x"]
    nev = c["nev"]
    with torch.cuda.stream(stream):
        if kind == "job":
            sec = g.build_sector_fields(ctx, L, s["fields"], nup=nup)
            g.solve_near_dev(sec, c["eps"], nev, s["evals"], s["evecs"], s["resid"], stream=stream, precision=PREC[c["prec"]])
        g.observables_dev(ctx, L, nev, s["evals"], s["evecs"], s["r"], s["r_mean"], s["s1p"], s["se"], stream=stream, nup=nup)
        if kind == "job":
            return {"evals": s["evals"], "evecs": _stored(s["evecs"]), "r": s["r"], "s1p": s["s1p"].float(), "se": s["se"].float()}
        g.observables_extra_dev(ctx, L, nev, s["evecs"], 2.0, s["kl"], s["sqp"], s["fluct"], s["dynf"], stream=stream, nup=nup)
    return {k: s[k] for k in ("r", "r_mean", "s1p", "se", "kl", "sqp", "fluct", "dynf")}


# ---- what a pass cannot do without ----------------------------------------------------------------------


def _sizes(c):
    """n, entries of H, and entries and flops of a sparse factor of H - sigma.  The last two grow as powers
    of n on this graph: 8.4e6 entries and 1.0e10 flops at n = 12870, 11.5 and 38 times that at n = 48620."""
    L, nup = c["L"], c["nup"]
    n = math.comb(L, nup)
    nnz = n + n * 2.0 * nup * (L - nup) / (L - 1)
    return n, nnz, 8.4e6 * (n / 12870) ** 1.84, 1.0e10 * (n / 12870) ** 2.74


def work(c):
    """The factor is written once and read twice (forward, backward) by one block solve; a job needs at least
    nev columns through it.  H is written once when the sector is built and read once by each product."""
    n, nnz, nl, fl = _sizes(c)
    kind = c["kind"]
    word = 8.0 if c.get("prec") == "fp64" else 4.0
    if kind == "bounds":  # E_min and E_max: about 2 L products, three vectors each
        k = 2 * c["L"]
        return {"bytes": 12 * nnz * (1 + k) + 24.0 * n * k, "flops": 2 * nnz * k}
    if kind == "observe":
        v = 8.0 * n * c["nev"]
        return {"bytes": 2 * v, "flops": 4.0 * n * c["nev"] * 2 ** (c["L"] / 2 - 1) / c["L"]}
    if kind == "solve":
        return {"bytes": 2 * nl * word + 12 * nnz + 16.0 * n * c["p"], "flops": 4 * nl * c["p"] + 2 * nnz * c["p"]}
    if kind == "factor":
        return {"bytes": 3 * nl * word + 24 * nnz + 16.0 * n * c["p"], "flops": fl + 4 * nl * c["p"] + 2 * nnz * c["p"]}
    blocks = -(-c["nev"] // 8)
    one = {"bytes": nl * word * (1 + 2 * blocks) + 12 * nnz * (1 + 2 * c["L"] + blocks) + 12.0 * n * c["nev"],
           "flops": fl + 4 * nl * c["nev"] + 2.0 * n * c["nev"] ** 2}
    k = c.get("jobs", 1)
    return {"bytes": k * one["bytes"], "flops": k * one["flops"]}


# ---- the same in plain torch, 64 bits -------------------------------------------------------------------


def _basis(L, nup):
    s = torch.arange(1 << L, device="cuda")
    bits = sum((s >> i) & 1 for i in range(L))
    return s[bits == nup]


def _hamiltonian(c, h):
    """Basis, and H = sum_i S_i.S_{i+1} + sum_i h_i S^z_i on it: diagonal, and (row, column) of the 1/2 entries."""
    L = c["L"]
    st = _basis(L, c["nup"])
    diag = torch.zeros(len(st), device="cuda", dtype=torch.float64)
    rows, cols = [], []
    for i in range(L):
        j = (i + 1) % L
        si, sj = (st >> i) & 1, (st >> j) & 1
        diag += torch.where(si == sj, 0.25, -0.25).double() + (si.double() - 0.5) * float(h[i])
        at = (si != sj).nonzero().flatten()
        rows.append(at)
        cols.append(torch.searchsorted(st, st[at] ^ ((1 << i) | (1 << j))))
    return st, diag, torch.cat(rows), torch.cat(cols)


def _dense(diag, rows, cols):
    H = torch.diag(diag)
    H[rows, cols] += 0.5
    return H


def _extremes(diag, rows, cols, steps=250):
    """E_min and E_max by Lanczos with full reorthogonalization."""
    n = len(diag)
    order = torch.argsort(rows)
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.bincount(rows, minlength=n).cumsum(0)
    A = torch.sparse_csr_tensor(ptr, cols[order], torch.full((len(rows),), 0.5, device="cuda", dtype=torch.float64), (n, n))
    steps = min(steps, n - 1)
    V = torch.zeros(steps, n, device="cuda", dtype=torch.float64)
    v, al, be = _normal((n,), 1), [], []
    for k in range(steps):
        b = v.norm()
        be.append(b)
        v = v / b
        V[k] = v
        w = diag * v + (A @ v[:, None])[:, 0]
        al.append(w @ v)
        for _ in range(2):
            w = w - V[: k + 1].T @ (V[: k + 1] @ w)
        v = w
    be = torch.stack(be[1:])
    T = torch.diag(torch.stack(al)) + torch.diag(be, 1) + torch.diag(be, -1)
    e = torch.linalg.eigvalsh(T.cpu())
    return float(e[0]), float(e[-1])


def _nearest(e, sigma, nev):
    return torch.argsort((e - sigma).abs(), stable=True)[:nev].sort().values


def _eigenpairs(c, h):
    """The nev eigenpairs nearest the target, ascending; vectors as rows."""
    _, diag, rows, cols = _hamiltonian(c, h)
    H = _dense(diag, rows, cols)
    n, nev = len(diag), c["nev"]
    if n <= 4000:
        e, V = torch.linalg.eigh(H)
        at = _nearest(e, float(e[0] + c["eps"] * (e[-1] - e[0])), nev)
        return e[at], V[:, at].T.contiguous()
    lo, hi = _extremes(diag, rows, cols)
    sigma = lo + c["eps"] * (hi - lo)
    lu = torch.linalg.lu_factor(H - sigma * torch.eye(n, device="cuda", dtype=torch.float64))
    p = 20
    X, V = _normal((n, p), 2), None
    for _ in range(6 + (5 * nev) // p):  # block Krylov space of (H - sigma)^-1, not restarted
        X = torch.linalg.lu_solve(*lu, X)
        for _ in range(3):
            if V is not None:
                X = X - V @ (V.T @ X)
            X = torch.linalg.qr(X)[0]
        V = X if V is None else torch.cat([V, X], 1)
    W = V.T @ torch.linalg.lu_solve(*lu, V)
    t, S = torch.linalg.eigh((W + W.T) / 2)
    V = torch.linalg.qr(V @ S[:, torch.argsort(t.abs(), descending=True)[: nev + 20]])[0]
    e, S = torch.linalg.eigh(V.T @ (H @ V))
    at = _nearest(e, sigma, nev)
    return e[at], (V @ S[:, at]).T.contiguous()


def _gap_ratios(e):
    d = e[1:] - e[:-1]
    return torch.minimum(d[:-1], d[1:]) / torch.maximum(d[:-1], d[1:])


def _xlogx(p):
    return torch.where(p > 0, p * torch.log(torch.where(p > 0, p, 1.0)), 0.0)


def _entropies(c, V):
    """Participation entropy S_1, and entanglement entropy of the first floor(L/2) sites."""
    st, half = _basis(c["L"], c["nup"]), c["L"] // 2
    P = V * V / (V * V).sum(1, keepdim=True)
    se = []
    for v in V:
        M = torch.zeros(1 << half, 1 << (c["L"] - half), device="cuda", dtype=torch.float64)
        M[st & ((1 << half) - 1), st >> half] = v / v.norm()
        w = torch.linalg.svdvals(M) ** 2
        se.append(-_xlogx(torch.where(w > 1e-15, w, 0.0)).sum())
    return -_xlogx(P).sum(1), torch.stack(se)


def _further(c, V):
    """Kullback-Leibler divergence of neighbours, S_2, variance of S^z of the half chain, dynamic fraction."""
    L = c["L"]
    st = _basis(L, c["nup"])
    P = V * V / (V * V).sum(1, keepdim=True)
    spin = torch.stack([((st >> i) & 1).double() - 0.5 for i in range(L)])
    half = spin[: L // 2].sum(0)
    kl = (P[:-1] * torch.log(P[:-1] / P[1:])).sum(1)
    mean = P @ half
    fluct = (P * (half - mean[:, None]) ** 2).sum(1)
    ang = 2 * math.pi * torch.arange(L, device="cuda", dtype=torch.float64) / L
    re, im = torch.cos(ang) @ spin, torch.sin(ang) @ spin
    dynf = 1 - ((P @ re) ** 2 + (P @ im) ** 2) / (P @ (re * re + im * im))
    return kl, -torch.log((P * P).sum(1)), fluct, dynf


def exact(c, seed):
    kind = c["kind"]
    n = math.comb(c["L"], c["nup"])
    if kind == "bounds":
        return list(_extremes(*_hamiltonian(c, _fields(c, seed))[1:]))
    if kind == "observe":
        V, e = _vectors(c, seed), _levels(c, seed)
        r = _gap_ratios(e)
        s1, se = _entropies(c, V)
        kl, s2, fluct, dynf = _further(c, V)
        return {"r": r, "r_mean": r.mean()[None], "s1p": s1, "se": se, "kl": kl, "sqp": s2, "fluct": fluct, "dynf": dynf}
    if n > 13000:  # the dense factorization would take too long
        return None
    if kind in ("factor", "solve"):
        _, diag, rows, cols = _hamiltonian(c, _fields(c, seed))
        sigma = _target(c, *_extremes(diag, rows, cols))
        A = _dense(diag - sigma, rows, cols)
        b = _normal((c["p"], n), seed).T
        lu = torch.linalg.lu_factor(A)
        x = torch.linalg.lu_solve(*lu, b)
        for _ in range(2):
            x = x + torch.linalg.lu_solve(*lu, b - A @ x)
        return x.T.contiguous()
    jobs = []
    for k in range(c["jobs"] if kind == "served" else 1):
        e, V = _eigenpairs(c, _fields(c, seed, k))
        s1, se = _entropies(c, V)
        jobs.append({"evals": e, "evecs": V, "r": _gap_ratios(e), "s1p": s1, "se": se})
    if kind == "served":
        return {k: torch.stack([j[k] for j in jobs]) for k in ("evals", "r", "s1p", "se")}
    return dict(jobs[0], evecs=_stored(jobs[0]["evecs"]).double() if n <= 4000 else None)
