"""Performance cases: the calls a user of this library makes, over the sizes they make them at.

A case is one pass through a public entry point of ``paper_2307_10675_gb300``:

* ``sigma``       ``ifci_sigma``: one H c of a CI space CAS(2m e, n o), any precision, vectors with
                  or without spin-flip symmetry (a user's own eigen-solver calls it in its loop);
* ``davidson``    ``ifci_davidson_batched``: a batch of 2-body CI problems;
* ``hbci``        ``ifci_hbci_batched``: a batch of 2-body problems by selected CI + PT2;
* ``increments``  ``ifci_increments``: a whole iFCI expansion;
* ``gradient``    ``ifci_rdm_backward``: its backward pass, on the vectors the forward call kept.

The integrals follow the recipe of the repository's synthetic chains (orbitals 1.5 Angstrom apart,
integrals that decay as exp(-d/2), Gaussian factors of rank 16), drawn here from the case's seed.
"""
from __future__ import annotations

import itertools
import math
import random

import numpy as np
import torch

import paper_2307_10675_gb300 as ifci

SPACING = 1.5
NAUX = 16
MAX_DETS = math.comb(20, 4) ** 2      # the largest space a case takes: CAS(8e,20o)
MAX_DETS_LOW = math.comb(18, 3) ** 2  # the same for the paths that keep every intermediate whole


def listed():
    return [
        # Smallest call: two 2-orbital bodies, 36 determinants; launches and host work are all of it.
        {"name": "sigma-4o-fp64", "kind": "sigma", "n": 4, "m": 2, "precision": "fp64", "sym": False},
        # A 2-body space of two 6-orbital bodies (4,356 determinants), the FP64-accurate tensor-core path
        # on a singlet (spin-flip-symmetric) vector: the commonest space of an expansion to 2 bodies.
        {"name": "sigma-12o-fp64e", "kind": "sigma", "n": 12, "m": 2, "precision": "fp64e", "sym": True},
        # Odd sizes and a vector without spin-flip symmetry (another solver's trial vector, a triplet).
        {"name": "sigma-15o-fp64e-general", "kind": "sigma", "n": 15, "m": 3, "precision": "fp64e", "sym": False},
        # The largest 3-body space of the 24- and 40-body chains: the hot loop of an expansion to 3 bodies.
        {"name": "sigma-18o-fp64e", "kind": "sigma", "n": 18, "m": 3, "precision": "fp64e", "sym": True},
        # A 4-body space, 2.3e7 determinants: more than 204 pairs, larger than one wave of intermediates.
        {"name": "sigma-20o-fp64e", "kind": "sigma", "n": 20, "m": 4, "precision": "fp64e", "sym": True},
        # The library's default precision on an odd 3-body space.
        {"name": "sigma-13o-fp64", "kind": "sigma", "n": 13, "m": 3, "precision": "fp64", "sym": False},
        # The low-precision contraction of the mixed solver's first phase.
        {"name": "sigma-17o-bf16", "kind": "sigma", "n": 17, "m": 3, "precision": "bf16", "sym": True},
        # 32 two-body problems of bodies of 2 to 6 orbitals in one batch, default options (FP64).
        {"name": "davidson-32x2body", "kind": "davidson", "count": 32, "lo": 2, "hi": 6, "precision": "fp64"},
        # Selected CI + PT2 at the paper's thresholds on a batch of two-body problems.
        {"name": "hbci-16x2body", "kind": "hbci", "count": 16, "lo": 3, "hi": 6, "precision": "fp64e"},
        # The small expansion a user tries first: four 2-orbital bodies to 2 bodies, default options.
        {"name": "increments-4x2", "kind": "increments", "nbody": 4, "lo": 2, "hi": 2, "order": 2,
         "precision": "fp64"},
        # An expansion to 3 bodies over uneven bodies of 2 to 6 orbitals (298 CI problems up to
        # 665,856 determinants, near and far apart): the benchmark's workload at a smaller body count.
        {"name": "increments-12", "kind": "increments", "nbody": 12, "lo": 2, "hi": 6, "order": 3,
         "precision": "fp64e"},
        # Backward pass of an expansion to 3 bodies (63 CI problems).
        {"name": "gradient-7", "kind": "gradient", "nbody": 7, "lo": 2, "hi": 4, "order": 3},
    ]


def draw(rng: random.Random):
    known = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        case = _draw(rng)
        if case not in known:
            return case


def _draw(rng):
    kind = rng.choices(["sigma", "davidson", "hbci", "increments", "gradient"], [12, 3, 2, 4, 2])[0]
    if kind == "sigma":
        precision = rng.choices(["fp64e", "fp64", "bf16", "tf32", "fp32"], [12, 5, 2, 1, 1])[0]
        cap = MAX_DETS if precision == "fp64e" else MAX_DETS_LOW
        top = {"fp64e": 24, "bf16": 22, "tf32": 22}.get(precision, 24)
        target = math.exp(rng.uniform(math.log(36.0), math.log(cap)))
        m = rng.choice([2, 2, 3, 3, 3, 4, 4, 5])
        fits = [n for n in range(m + 2, top + 1)
                if math.comb(n, m) ** 2 <= cap and math.comb(n, m) ** 2 * n * (n + 1) <= MAX_DETS * 420]
        n = min(fits, key=lambda k: abs(math.log(math.comb(k, m) ** 2 / target)))
        return {"kind": kind, "n": n, "m": m, "precision": precision, "sym": rng.random() < 0.6}
    if kind == "davidson":
        count = round(math.exp(rng.uniform(0.0, math.log(96.0))))
        hi = rng.randint(3, 6)
        return {"kind": kind, "count": count, "lo": rng.randint(2, hi), "hi": hi,
                "precision": rng.choice(["fp64", "fp64e", "fp64e", "bf16"])}
    if kind == "hbci":
        hi = rng.randint(3, 6)
        return {"kind": kind, "count": round(math.exp(rng.uniform(0.0, math.log(24.0)))), "lo": rng.randint(2, hi),
                "hi": hi, "precision": "fp64e"}
    if kind == "increments":
        order = rng.choice([2, 3, 3])
        nbody = rng.randint(4, 11) if order == 3 else rng.randint(4, 24)
        hi = rng.randint(3, 6)
        return {"kind": kind, "nbody": nbody, "lo": 2, "hi": hi, "order": order,
                "precision": "fp64e" if order == 3 else rng.choice(["fp64", "fp64e"])}
    return {"kind": kind, "nbody": rng.randint(4, 8), "lo": 2, "hi": rng.randint(3, 4), "order": rng.randint(2, 3)}


# ---------------------------------------------------------------- inputs

def _rng(case, seed):
    return np.random.Generator(np.random.PCG64([int(seed) & 0xFFFFFFFF, 20]))


def _pairs(n):
    P, Q = np.tril_indices(n)
    return P, Q


def _chain(sizes, rng):
    """(h (norb, norb), V (npair, npair)) of a chain of bodies, float64 on the GPU."""
    norb = sum(sizes)
    x = SPACING * np.arange(norb)
    d = np.abs(x[:, None] - x[None, :])
    bonding = np.zeros(norb, dtype=bool)
    bonding[np.cumsum([0] + list(sizes[:-1]))] = True
    h = -0.3 * np.exp(-d / 2.0)
    h[np.arange(norb), np.arange(norb)] = np.where(bonding, -1.0, 0.5) + 0.3 * rng.normal(size=norb)
    P, Q = _pairs(norb)
    b = 0.1 * rng.normal(size=(NAUX, P.size)) * np.exp(-d[P, Q] / 2.0)
    b = torch.tensor(b, device="cuda")
    return torch.tensor(h, device="cuda"), (b.T @ b).contiguous()


def _sizes(case):
    """Body sizes of a case: lo..hi in turn, in an order that is a function of the case alone."""
    lo, hi = case["lo"], case["hi"]
    sizes = [lo + i % (hi - lo + 1) for i in range(case["nbody"])][::-1]
    random.Random(case["nbody"]).shuffle(sizes)
    return sizes


def _space_sizes(case, i):
    lo, hi = case["lo"], case["hi"]
    w = hi - lo + 1
    return [hi - i % w, lo + (i // w) % w]


def _split(n, m):
    return [n // m + (1 if i < n % m else 0) for i in range(m)]


_HANDLE = None


def _handle():
    """One handle for the program, as a user's program keeps one."""
    global _HANDLE
    if _HANDLE is None:
        _HANDLE = ifci.Handle(0, 0)
    return _HANDLE


def prepare(case, seed):
    rng = _rng(case, seed)
    kind = case["kind"]
    if kind == "sigma":
        h, V = _chain(_split(case["n"], case["m"]), rng)
        handle = _handle()
        tables = ifci.ifci_build_strings(handle, case["n"], case["m"])
        return {"kind": kind, "handle": handle, "tables": tables, "h": h, "V": V,
                "c": _vector(case, tables.nstr, seed).reshape(-1),
                "precision": ifci.PRECISIONS[case["precision"]], "sym": case["sym"]}
    if kind in ("davidson", "hbci"):
        problems, starts = [], []
        for i in range(case["count"]):
            sizes = _space_sizes(case, i)
            h, V = _chain(sizes, rng)
            problems.append(ifci.CIProblem(sum(sizes), 2, h, V, 0.0))
            starts.append(ifci.reference_determinant(sizes, (0, 1)))
        return {"kind": kind, "handle": _handle(), "problems": problems, "starts": starts,
                "opts": ifci.davidson_opts(case["precision"])}
    sizes = _sizes(case)
    h, V = _chain(sizes, rng)
    system = ifci.SystemArrays(np.cumsum([0] + sizes), h, V)
    if kind == "increments":
        return {"kind": kind, "handle": _handle(), "system": system, "order": case["order"],
                "opts": ifci.davidson_opts(case["precision"])}
    # the forward call keeps its vectors in the handle (one handle per state), tightly converged as gradients want
    handle = ifci.Handle(0, 0)
    opts = ifci.davidson_opts("fp64", r_tol=1e-10, max_iter=300)
    ifci.ifci_increments(handle, system, case["order"], opts)
    return {"kind": kind, "handle": handle, "system": system, "order": case["order"], "opts": opts}


def _vector(case, nstr, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    c = torch.randn((nstr, nstr), generator=g, device="cuda", dtype=torch.float64)
    if case["sym"]:
        c = 0.5 * (c + c.T)
    return (c / c.norm()).contiguous()


# ---------------------------------------------------------------- one pass

def run(state):
    kind, handle = state["kind"], state["handle"]
    if kind == "sigma":
        return ifci.ifci_sigma(handle, state["tables"], state["h"], state["V"], state["c"],
                               precision=state["precision"], spin_symmetric=state["sym"])
    if kind == "davidson":
        # (energies, sigma builds, status): the middle one counts work, it is no result
        e, _, status = ifci.ifci_davidson_batched(handle, state["problems"], state["opts"])
        return {"energies": e, "status": status}
    if kind == "hbci":
        out = ifci.ifci_hbci_batched(handle, state["problems"], state["starts"], opts=state["opts"])
        return {k: out[k] for k in ("e_var", "e_pt2", "nsel", "status")}
    if kind == "increments":
        out = ifci.ifci_increments(handle, state["system"], state["order"], state["opts"])
        return {k: out[k] for k in ("e0", "e_x", "eps", "e_total", "status")}
    dh, dV = ifci.ifci_rdm_backward(handle, state["system"], state["order"], 1.0, state["opts"])
    return {"dh": dh, "dV": dV}


# ---------------------------------------------------------------- work

def _space_work(n, m, builds, vectors):
    """Bytes and operations of `builds` products H c (the nonzero elements of H once each, c read and
    H c written) and of `vectors` more reads or writes of a vector."""
    ndet = math.comb(n, m) ** 2
    npair = n * (n + 1) // 2
    ns, nd = m * (n - m), math.comb(m, 2) * math.comb(n - m, 2)
    row = 1 + 2 * ns + 2 * nd + ns * ns
    return {"bytes": 8.0 * (npair * npair + n * n) + 8.0 * ndet * (2 * builds + vectors),
            "flops": 2.0 * ndet * row * builds}


def _sum(parts):
    parts = list(parts)
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


def work(case):
    kind = case["kind"]
    if kind == "sigma":
        return _space_work(case["n"], case["m"], 1, 0)
    # a solve cannot do without about ten products and, with each, two passes over a vector
    if kind in ("davidson", "hbci"):
        return _sum(_space_work(sum(_space_sizes(case, i)), 2, 10, 20) for i in range(case["count"]))
    sizes = _sizes(case)
    sets = [X for k in range(1, case["order"] + 1) for X in itertools.combinations(range(len(sizes)), k)]
    norb = sum(sizes)
    npair = norb * (norb + 1) // 2
    if kind == "increments":
        w = _sum(_space_work(sum(sizes[b] for b in X), len(X), 10, 20) for X in sets)
        w["bytes"] += 8.0 * npair * npair
        return w
    # moments of every vector: each pair of single excitations of a determinant once
    w = {"bytes": 8.0 * npair * npair, "flops": 0.0}
    for X in sets:
        n, m = sum(sizes[b] for b in X), len(X)
        ndet = math.comb(n, m) ** 2
        w["bytes"] += 8.0 * ndet
        w["flops"] += 2.0 * ndet * (2 * m * (n - m + 1)) ** 2 / 2
    return w


# ---------------------------------------------------------------- the same in plain torch, 64 bits

def _tables(n, m):
    """J (npair, nstr) and s (npair, nstr): (E_pq + E_qp) |I> = s |J>, E_pp for p = q; s = 0 where there is none."""
    strs = sorted(sum(1 << p for p in occ) for occ in itertools.combinations(range(n), m))
    mask = np.array(strs, dtype=np.int64)
    P, Q = _pairs(n)
    J = np.zeros((P.size, mask.size), dtype=np.int64)
    s = np.zeros((P.size, mask.size))
    for a, (p, q) in enumerate(zip(P, Q)):
        op, oq = (mask >> p) & 1, (mask >> q) & 1
        if p == q:
            J[a], s[a] = np.arange(mask.size), op
            continue
        moved = np.where(op != oq, mask ^ (1 << int(p)) ^ (1 << int(q)), mask)
        J[a] = np.searchsorted(mask, moved)
        between = mask & (((1 << int(p)) - 1) & ~((2 << int(q)) - 1))
        odd = np.zeros(mask.size, dtype=np.int64)
        for r in range(n):
            odd ^= (between >> r) & 1
        s[a] = np.where(op != oq, 1.0 - 2.0 * odd, 0.0)
    return torch.tensor(J, device="cuda"), torch.tensor(s, device="cuda")


def _folded(h, V, nelec):
    """W with H c = sum_AB E_A W_AB (E_B c): the one-electron part folded in by sum_r E_rr = nelec."""
    n = h.shape[0]
    P, Q = (torch.tensor(v, device="cuda") for v in _pairs(n))
    r = torch.arange(n, device="cuda")

    def pair(p, q):
        hi, lo = torch.maximum(p, q), torch.minimum(p, q)
        return hi * (hi + 1) // 2 + lo

    ex = V[pair(P[:, None], r[None, :]), pair(r[None, :], Q[:, None])].sum(1)
    k = 0.5 * (h[P, Q] + h[Q, P]) - 0.5 * ex
    d = (P == Q).to(h.dtype)
    return 0.5 * (0.5 * (V + V.T) + (k[:, None] * d[None, :] + d[:, None] * k[None, :]) / nelec)


def _hc(W, J, s, C):
    """H C of an (nstr, nstr) coefficient matrix."""
    npair, nstr = J.shape
    if npair * nstr * nstr <= 1 << 27:
        D = s[:, :, None] * C[J] + (s[:, :, None] * C.T[J]).transpose(1, 2)
        G = torch.tensordot(W, D, dims=1)
        G = s[:, :, None] * torch.gather(G, 1, J[:, :, None].expand_as(G)) + \
            s[:, None, :] * torch.gather(G, 2, J[:, None, :].expand_as(G))
        return G.sum(0)
    D = torch.empty((npair, nstr, nstr), dtype=C.dtype, device=C.device)
    for a in range(npair):
        D[a] = s[a][:, None] * C[J[a]] + s[a][None, :] * C[:, J[a]]
    G = (W @ D.reshape(npair, -1)).reshape(npair, nstr, nstr)
    out = torch.zeros_like(C)
    for a in range(npair):
        out += s[a][:, None] * G[a][J[a]] + s[a][None, :] * G[a][:, J[a]]
    return out


def _lowest(h, V, m):
    """Lowest eigenpair of H among the symmetric coefficient matrices (Lanczos, every vector kept)."""
    n = h.shape[0]
    J, s = _tables(n, m)
    W = _folded(h, V, 2 * m)
    nstr = J.shape[1]
    dim = nstr * (nstr + 1) // 2
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    v = torch.randn((nstr, nstr), generator=g, device="cuda", dtype=torch.float64)
    v = v + v.T
    basis, alpha, beta = [(v / v.norm()).reshape(-1)], [], []
    best = None
    for k in range(min(dim, 400)):
        w = _hc(W, J, s, basis[k].reshape(nstr, nstr)).reshape(-1)
        alpha.append(float(w @ basis[k]))
        B = torch.stack(basis)
        for _ in range(2):
            w = w - B.T @ (B @ w)
        beta.append(float(w.norm()))
        done = beta[-1] < 1e-12 or k + 1 == min(dim, 400)
        if k % 10 == 9 or done:
            T = np.diag(alpha) + np.diag(beta[:-1], 1) + np.diag(beta[:-1], -1)
            e, y = np.linalg.eigh(T)
            best = (e[0], B.T @ torch.tensor(y[:, 0], device="cuda"))
            if done or abs(beta[-1] * y[-1, 0]) < 1e-12:
                break
        basis.append(w / beta[-1])
    x = best[1].reshape(nstr, nstr)
    return best[0], x, J, s


def _frozen(h, V, sizes, X):
    """(h1, V_X, e_core) of body set X: the other bodies' first orbitals doubly occupied, the rest removed."""
    off = np.cumsum([0] + sizes)
    act = np.concatenate([np.arange(off[b], off[b + 1]) for b in X]) if X else np.zeros(0, dtype=int)
    core = np.array([off[b] for b in range(len(sizes)) if b not in X], dtype=int)

    def pair(p, q):
        hi, lo = np.maximum(p, q), np.minimum(p, q)
        return hi * (hi + 1) // 2 + lo

    c, d = core[:, None], core[None, :]
    ec = 2.0 * h[core, core].sum() + (2.0 * V[pair(c, c), pair(d, d)] - V[pair(c, d), pair(d, c)]).sum()
    p, q, k = act[:, None, None], act[None, :, None], core[None, None, :]
    h1 = h[act[:, None], act[None, :]] + (2.0 * V[pair(p, q), pair(k, k)] - V[pair(p, k), pair(k, q)]).sum(-1)
    P, Q = _pairs(act.size)
    A = pair(act[P], act[Q])
    return h1, V[A[:, None], A[None, :]], ec


def exact(case, seed):
    rng = _rng(case, seed)
    kind = case["kind"]
    if kind == "sigma":
        n, m = case["n"], case["m"]
        h, V = _chain(_split(n, m), rng)
        J, s = _tables(n, m)
        C = _vector(case, J.shape[1], seed)
        return _hc(_folded(h, V, 2 * m), J, s, C).reshape(-1)
    if kind == "hbci":
        return None
    if kind == "davidson":
        if case["count"] > 48:
            return None
        e = []
        for i in range(case["count"]):
            h, V = _chain(_space_sizes(case, i), rng)
            e.append(_lowest(h, V, 2)[0])
        return {"energies": np.array(e), "status": None}
    sizes = _sizes(case)
    order = case["order"]
    sets = [X for k in range(1, order + 1) for X in itertools.combinations(range(len(sizes)), k)]
    cost = sum(math.comb(sum(sizes[b] for b in X), len(X)) ** 2 for X in sets)
    if cost > 1_500_000 or len(sets) > 120:
        return None
    h, V = _chain(sizes, rng)
    e0 = float(_frozen(h, V, sizes, ())[2])
    if kind == "increments":
        ex = {}
        for X in sets:
            h1, v, ec = _frozen(h, V, sizes, X)
            ex[X] = _lowest(h1, v, len(X))[0] + float(ec)
        eps = {}
        for X in sets:
            eps[X] = ex[X] - e0 - sum(eps[Y] for k in range(1, len(X)) for Y in itertools.combinations(X, k))
        return {"e0": e0, "e_x": np.array([ex[X] for X in sets]), "eps": np.array([eps[X] for X in sets]),
                "e_total": e0 + math.fsum(eps.values()), "status": None}
    # E = (1 - sum w) E_0 + sum_Y w_Y E_Y, each E_Y differentiated at its fixed vector (Hellmann-Feynman)
    h.requires_grad_(True)
    V.requires_grad_(True)
    N, wsum = len(sizes), 0.0
    for X in sets:
        k = len(X)
        w = 1.0 if k == N else (-1.0) ** (order - k) * math.comb(N - k - 1, order - k)
        wsum += w
        h1, v, ec = _frozen(h, V, sizes, X)
        _, x, J, s = _lowest(h1.detach(), v.detach(), k)
        (w * ((x * _hc(_folded(h1, v, 2 * k), J, s, x)).sum() + ec)).backward()
    ((1.0 - wsum) * _frozen(h, V, sizes, ())[2]).backward()
    return {"dh": 0.5 * (h.grad + h.grad.T), "dV": 0.5 * (V.grad + V.grad.T)}
