"""The work that a program has this framework do, as cases that can be timed.

Each case is one pass through the public entry points of ``paper_1910_03527_gb300``:
many-body expansions over batches of small tuple CASCIs (warp solver), of larger
ones (block solver) and of active spaces routed to the single-CAS solver, the
adjoint of the expansion energy, the screened expansion, and one large CAS (its
sigma product and its lowest state).  Inputs are the synthetic systems of
``workloads``: the half-filled Hubbard ring (momentum or Pipek-Mezey orbitals) and
the low-rank-ERI molecule, with couplings that the seed varies by a few percent.
"""

from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

import paper_1910_03527_gb300 as eng
from workloads import hubbard_ring_momentum, hubbard_ring_pm, synthetic_molecule


def _ring(name, task, L, max_order, precision, U=4.0, skip=True, basis="momentum"):
    return dict(name=name, task=task, system="ring", norb=L, U=U, basis=basis, max_order=max_order,
                skip=skip, precision=precision)


def _molecule(name, task, norb, max_order, precision):
    return dict(name=name, task=task, system="molecule", norb=norb, max_order=max_order, skip=False,
                precision=precision)


def listed():
    return [
        # The smallest expansion: the 8-site ring to full order in float64, no tuple
        # skipped. 255 CASCIs in eight orders; launches, small grids and the one
        # full-space CASCI at the end set its time.
        _ring("ring8_full_fp64", "mbe", 8, 8, "fp64", U=2.0, skip=False),
        # The headline expansion: 107,085 CASCIs of 2-6 orbitals (at most 400
        # determinants), mixed precision and float64.
        _ring("ring22_o6_mixed", "mbe", 22, 6, "mixed"),
        _ring("ring22_o6_fp64", "mbe", 22, 6, "fp64"),
        # A screened expansion: spawned children, sorted lists of a million tuples.
        _ring("ring46_screened_o5_mixed", "screened", 46, 5, "mixed"),
        # Energy and its derivatives with respect to every integral: the orders 1-4 of
        # the 46-site ring, float64, forward and backward.
        _ring("ring46_adjoint_o4_fp64", "adjoint", 46, 4, "fp64"),
        # Molecular tuples on a (6e,6o) reference space: 595 CASCIs of 7 and 8
        # orbitals (up to 4,900 determinants), and 469 of 7-9 (up to 15,876).
        _molecule("molecule40_o2_mixed", "mbe", 40, 2, "mixed"),
        _molecule("molecule20_o3_mixed", "mbe", 20, 3, "mixed"),
        # Derivatives of the molecular expansion, float64.
        _molecule("molecule20_adjoint_o2_fp64", "adjoint", 20, 2, "fp64"),
        # A Type-2 expansion: reference space of all 13 occupied orbitals, tuple spaces
        # of 14 and 15 orbitals, each routed to the single-CAS solver.
        dict(name="ring26_type2_o2_mixed", task="type2", system="ring", norb=26, U=4.0, basis="momentum",
             max_order=2, skip=True, precision="mixed"),
        # One large CAS of the molecule: sigma of 12 orbitals in float64 (853,776
        # determinants) and of 14 in float32 (11,778,624), and the lowest state of 12.
        dict(name="sigma12_fp64", task="sigma", system="molecule", norb=40, n_cas=12, precision="fp64"),
        dict(name="sigma14_mixed", task="sigma", system="molecule", norb=40, n_cas=14, precision="mixed"),
        dict(name="solve12_mixed", task="solve", system="molecule", norb=40, n_cas=12, precision="mixed"),
    ]


# Largest passes that draw() gives, in tuples of one expansion (by the listed cases).
_MAX_TUPLES = {("mbe", "ring"): 107085, ("adjoint", "ring"): 157642, ("screened", "ring"): 1400000,
               ("mbe", "molecule"): 595, ("adjoint", "molecule"): 105}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        task = rng.choice(["mbe", "mbe", "mbe", "screened", "adjoint", "type2", "sigma", "solve"])
        precision = rng.choice(["mixed", "fp64"])
        if task in ("sigma", "solve"):
            # (the largest spaces in mixed precision only: a float64 pass over them takes longer)
            top = {"sigma": (13, 14), "solve": (11, 12)}[task][precision == "mixed"]
            return dict(task=task, system="molecule", norb=rng.randint(18, 40), n_cas=rng.randint(8, top),
                        precision=precision)
        if task == "type2":
            # (tuple spaces of 7-11 orbitals: batched; of 14-16: routed)
            return dict(task=task, system="ring", norb=rng.choice([12, 14, 16, 18, 26, 28]), U=round(rng.uniform(1.0, 6.0), 2),
                        basis="momentum", max_order=rng.randint(1, 2), skip=True, precision="mixed")
        if task == "screened" or rng.random() < 0.6:
            lo, hi = {"mbe": (8, 22), "adjoint": (10, 46), "screened": (16, 46)}[task]
            case = dict(task=task, system="ring", norb=_log_int(rng, lo, hi), U=round(rng.uniform(1.0, 6.0), 2),
                        basis=rng.choice(["momentum", "pm"]), max_order=rng.randint(3, 6), skip=True,
                        precision="fp64" if task == "adjoint" else precision)
            if task == "screened":
                case["max_order"] = rng.randint(3, 5)
            if task == "adjoint":  # closed-shell rings (4 m + 2 sites): their ground states are not degenerate
                case.update(norb=4 * ((case["norb"] - 2) // 4) + 2, max_order=rng.randint(3, 4))
        else:
            case = dict(task=task, system="molecule", norb=rng.randint(12, 40), max_order=rng.randint(1, 3),
                        skip=False, precision="fp64" if task == "adjoint" else precision)
            if task == "adjoint" or precision == "fp64":
                case["max_order"] = min(case["max_order"], 2)
        count = sum(c for o in _tuple_counts(case).values() for c in o.values())
        if count <= _MAX_TUPLES[(task, case["system"])]:
            return case


# ------------------------------------------------------------------ inputs

_MOL_REF = list(range(5, 11))  # the (6e,6o) reference space around the Fermi level


@functools.lru_cache(maxsize=16)
def _ring_unit(L, basis):
    """The ring's integrals at t = U = 1 (kept, since localising 46 orbitals takes a second)."""
    build = {"momentum": hubbard_ring_momentum, "pm": hubbard_ring_pm}[basis]
    h1, eri, occ, _ = build(L, 1.0, 1.0)
    return h1, eri, occ


def _integrals(case, seed):
    """h1, (pq|rs) and occupation of the case's system, its couplings varied by the seed."""
    rng = np.random.default_rng(seed)
    n = case["norb"]
    if case["system"] == "ring":
        h1, eri, occ = _ring_unit(n, case["basis"])
        t, U = 1.0 + 0.02 * rng.uniform(-1, 1), case["U"] * (1.0 + 0.05 * rng.uniform(-1, 1))
        return t * h1, U * eri, occ
    h1, eri, occ = synthetic_molecule(1910)
    noise = np.triu(rng.normal(0.0, 0.01, size=h1.shape), 1)
    h1, eri = h1 + noise + noise.T, eri * (1.0 + 0.02 * rng.uniform(-1, 1))
    return np.ascontiguousarray(h1[:n, :n]), np.ascontiguousarray(eri[:n, :n, :n, :n]), occ[:n].copy()


def _spaces(case, occ):
    n = case["norb"]
    if case["task"] == "type2":
        return eng.expansion_spaces(occ.tolist(), "type2")
    if case["system"] == "ring":
        return [], list(range(n))
    return _MOL_REF, [p for p in range(n) if p not in _MOL_REF]


def _cas(case):
    """The molecule's active space of n_cas orbitals around the Fermi level (orbitals 7 and 8)."""
    half = case["n_cas"] // 2
    lo = max(0, 8 - half)
    return list(range(lo, lo + case["n_cas"]))


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    h1, eri, occ = _integrals(case, seed)
    # gradients are taken to a residual of 1e-12 (their errors are of first order in the
    # residual, and the adjoint weights amplify them); energies to the default, one large
    # CAS to 1e-8
    tol = {"adjoint": 1e-12, "solve": 1e-8}.get(case["task"])
    opts = eng.Opts(precision=case["precision"], **({} if tol is None else {"tol": tol}))
    st = dict(case=case, ctx=eng.Context(0), opts=opts, occ_host=occ.tolist(),
              h1=torch.tensor(h1, device=dev), eri=torch.tensor(eri, device=dev), occ=torch.tensor(occ, device=dev))
    if case["task"] in ("sigma", "solve"):
        st["cas"] = _cas(case)
        if case["task"] == "sigma":
            st["c"] = _vector(case, occ, seed)
    else:
        st["ref"], st["exp"] = _spaces(case, occ)
        st["orders"] = list(range(1, case["max_order"] + 1))
    if case["task"] == "adjoint":
        st["h1"].requires_grad_(True)
        st["eri"].requires_grad_(True)
    return st


def _vector(case, occ, seed):
    """A unit CI vector: normal elements, as a correction vector of the Davidson has them."""
    ns = math.comb(case["n_cas"], int(sum(occ[p] for p in _cas(case))))
    g = torch.Generator(device="cuda").manual_seed(seed)
    c = torch.randn(ns * ns, generator=g, dtype=torch.float64, device="cuda")
    return c / c.norm()


# ------------------------------------------------------------------ one pass

def run(st):
    task = st["case"]["task"]
    if task == "sigma":
        sigma, _ = st["ctx"].casci_sigma_large(st["h1"], st["eri"], st["occ"], st["cas"], st["c"],
                                               precision=st["case"]["precision"])
        return sigma
    if task == "solve":
        # (the result also carries the residual reached and the products spent)
        r = st["ctx"].casci_solve(st["h1"], st["eri"], st["occ"], st["cas"], st["opts"])
        return dict(lam=r["lam"], eps=r["eps"], status=r["status"])
    if task == "adjoint":
        st["h1"].grad = st["eri"].grad = None
        e = eng.MBEEnergy.apply(st["h1"], st["eri"], st["ctx"], st["occ"], st["ref"], st["exp"], st["orders"],
                                st["case"]["skip"], st["opts"], True)
        e.backward()
        return dict(e_total=e.detach(), grad_h1=st["h1"].grad, grad_eri=st["eri"].grad)
    if task == "screened":
        out = eng.run_mbe_screened(st["ctx"], st["h1"], st["eri"], st["occ"], st["ref"], st["exp"],
                                   st["case"]["max_order"], st["case"]["skip"], opts=st["opts"],
                                   occ_host=st["occ_host"])
    else:
        out = eng.run_mbe(st["ctx"], st["h1"], st["eri"], st["occ"], st["ref"], st["exp"], st["orders"],
                          st["case"]["skip"], st["opts"], occ_host=st["occ_host"])
    # (out["iters"] records the sigma products that were spent, not a result)
    return {key: out[key] for key in ("tuples", "eps", "status", "inc", "e_order", "e_phi", "e_total")}


# ------------------------------------------------------------------ work

def _tuple_counts(case):
    """{order: {electron pairs k: tuples}} of a complete expansion, skip rule applied."""
    n = case["norb"]
    occ = n // 2 if case["system"] == "ring" else 8
    if case["task"] == "type2":
        ref_o, ref_v, xo, xv = occ, 0, 0, n - occ
    elif case["system"] == "ring":
        ref_o, ref_v, xo, xv = 0, 0, occ, n - occ
    else:
        ref_o, ref_v, xo, xv = 3, 3, occ - 3, n - occ - 3
    got = {}
    for m in range(1, case["max_order"] + 1):
        got[m] = {}
        for j in range(0, m + 1):
            c = math.comb(xo, j) * math.comb(xv, m - j)
            if c and not (case["skip"] and (ref_o + j == 0 or ref_v + m - j == 0)):
                got[m][ref_o + j] = c
    return got


def _sigma_flops(n, k, half):
    """One sigma product by the string-driven form: the opposite-spin double loop over the
    k (n - k + 1) replacements of each spin and the two same-spin products with the
    connected strings, on every determinant or (half) on one of each spin-flip pair."""
    ns = math.comb(n, k)
    conn = 1 + k * (n - k) + math.comb(k, 2) * math.comb(n - k, 2)
    dets = ns * (ns + 1) // 2 if half else ns * ns
    return dets * 2 * (2 * conn + (k * (n - k + 1)) ** 2)


# Sigma products that an iterative eigensolver needs on these Hamiltonians to the residuals
# asked for (the rings' states are dominated by one determinant, the molecule's are not).
_PRODUCTS = {"ring": 10, "molecule": 100}


def work(case):
    n = case["norb"]
    read = 8 * (n * n + n ** 4) + n
    if case["task"] in ("sigma", "solve"):
        m = case["n_cas"]
        k = 8 - max(0, 8 - m // 2)
        dets = math.comb(m, k) ** 2
        if case["task"] == "sigma":
            return dict(bytes=read + 16 * dets, flops=_sigma_flops(m, k, False))
        return dict(bytes=read + 8 * dets, flops=2 * _PRODUCTS["molecule"] * _sigma_flops(m, k, True))
    ref = {"type2": n // 2}.get(case["task"], 0 if case["system"] == "ring" else 6)
    flops, written = 0, 0
    for m, by_k in _tuple_counts(case).items():
        written += sum(by_k.values()) * (4 * m + 8 + 4 + 8)
        flops += sum(c * _PRODUCTS[case["system"]] * _sigma_flops(ref + m, k, True) for k, c in by_k.items())
    if case["task"] == "adjoint":
        written = 8 * (n * n + n ** 4)
    return dict(bytes=read + written, flops=flops)


# ------------------------------------------------------------------ plain 64-bit reference

@functools.lru_cache(maxsize=64)
def _strings(n, k):
    return sorted(sum(1 << p for p in c) for c in itertools.combinations(range(n), k))


@functools.lru_cache(maxsize=64)
def _replacements(n, k):
    """E_pq |J> = sign |I> on the strings of k electrons in n orbitals, as
    {(p, q): (I, J, sign) index lists}."""
    strings = _strings(n, k)
    at = {s: i for i, s in enumerate(strings)}
    ops = {(p, q): ([], [], []) for p in range(n) for q in range(n)}
    for j, s in enumerate(strings):
        for q in range(n):
            if not s >> q & 1:
                continue
            for p in range(n):
                r = s & ~(1 << q)
                if r >> p & 1:
                    continue
                between = bin(r & ((1 << max(p, q)) - 1) & ~((1 << (min(p, q) + 1)) - 1)).count("1")
                for lst, v in zip(ops[(p, q)], (at[r | 1 << p], j, (-1.0) ** between)):
                    lst.append(v)
    return ops


@functools.lru_cache(maxsize=64)
def _dense_ops(n, k, device):
    """E_pq as dense matrices [n, n, Ns, Ns]."""
    ns = math.comb(n, k)
    e = torch.zeros((n, n, ns, ns), dtype=torch.float64, device=device)
    for (p, q), (i, j, s) in _replacements(n, k).items():
        if i:
            e[p, q, i, j] = torch.tensor(s, dtype=torch.float64, device=device)
    return e


def _active(h1, eri, occ, A):
    """One-electron operator in the frozen core's field, active integrals, and the core's
    energy, of active orbitals A [T, n] (two-electron terms symmetric in the two pairs)."""
    n = A.shape[1]
    act = torch.zeros((A.shape[0], h1.shape[0]), dtype=torch.bool, device=h1.device)
    act.scatter_(1, A, True)
    core = (occ.bool()[None, :] & ~act).double()
    j = torch.einsum("pqcc->cpq", eri) + torch.einsum("ccpq->cpq", eri)
    k = 0.5 * (torch.einsum("cqpc->cpq", eri) + torch.einsum("pccq->cpq", eri))
    f = h1[None] + torch.einsum("tc,cpq->tpq", core, j - k)
    h = torch.gather(torch.gather(f, 1, A[:, :, None].expand(-1, -1, h1.shape[0])), 2, A[:, None, :].expand(-1, n, -1))
    g = eri[A[:, :, None, None, None], A[:, None, :, None, None], A[:, None, None, :, None], A[:, None, None, None, :]]
    jk = 2.0 * torch.einsum("iijj->ij", eri) - torch.einsum("ijji->ij", eri)
    e_core = 2.0 * core @ torch.diagonal(h1) + torch.einsum("ti,tj,ij->t", core, core, jk)
    return h, g, e_core


def _string_hamiltonian(h, g, e):
    """One-spin part: sum h_pq E_pq + 1/2 sum (pq|rs) (E_pq E_rs - d_qr E_ps)."""
    hp = h - 0.5 * torch.einsum("tprrs->tps", g)
    n, ns = e.shape[0], e.shape[2]
    x = torch.einsum("tpqrs,rskj->tpqkj", g, e)
    return torch.einsum("tpq,pqij->tij", hp, e) + 0.5 * torch.einsum("pqik,tpqkj->tij", e, x.reshape(-1, n, n, ns, ns))


def _sector_bases(ns, device):
    """Orthonormal bases of the even and the odd states under exchange of the two spins."""
    ia, ib = torch.triu_indices(ns, ns, 0, device=device)
    even = torch.zeros((ns * ns, ia.numel()), dtype=torch.float64, device=device)
    c = torch.full((ia.numel(),), math.sqrt(0.5), dtype=torch.float64, device=device).masked_fill(ia == ib, 1.0)
    r = torch.arange(ia.numel(), device=device)
    even[ia * ns + ib, r] = c
    even[ib * ns + ia, r] = c
    ia, ib = torch.triu_indices(ns, ns, 1, device=device)
    odd = torch.zeros((ns * ns, ia.numel()), dtype=torch.float64, device=device)
    r = torch.arange(ia.numel(), device=device)
    odd[ia * ns + ib, r] = math.sqrt(0.5)
    odd[ib * ns + ia, r] = -math.sqrt(0.5)
    return [even, odd]


def _lowest(h1, eri, occ, A, k):
    """Total energies E_CAS(A) of active orbitals A [T, n], all with k electron pairs."""
    n, dev = A.shape[1], h1.device
    h, g, e_core = _active(h1, eri, occ, A)
    if k in (0, n):
        d = torch.arange(n, device=dev)
        jk = 2.0 * g[:, d[:, None], d[:, None], d[None, :], d[None, :]] - g[:, d[:, None], d[None, :], d[None, :], d[:, None]]
        full = 2.0 * h[:, d, d].sum(1) + jk.sum((1, 2))
        return e_core + (full if k else 0.0)
    e = _dense_ops(n, k, str(dev))
    ns = e.shape[2]
    hs = _string_hamiltonian(h, g, e)
    x = torch.einsum("tpqrs,rsij->tpqij", 0.5 * (g + g.permute(0, 3, 4, 1, 2)), e)
    one = torch.eye(ns, dtype=torch.float64, device=dev)
    H = torch.einsum("pqik,tpqjl->tijkl", e, x) + torch.einsum("tik,jl->tijkl", hs, one) + \
        torch.einsum("ik,tjl->tijkl", one, hs)
    H = H.reshape(-1, ns * ns, ns * ns)
    H = 0.5 * (H + H.transpose(1, 2))
    low = [torch.linalg.eigvalsh(b.T @ H @ b)[:, 0] for b in _sector_bases(ns, dev) if b.shape[1]]
    return e_core + (low[0] if len(low) == 1 else torch.minimum(*low))


def _chunks(A, k):
    dets = math.comb(A.shape[1], k) ** 2
    return A.split(max(1, 60_000_000 // (dets * dets)))


def _expansion(h1, eri, occ, ref, exp, orders, skip):
    """Per order: (tuples, eps, increments), and E_Phi and the total, by definition."""
    occ_l = occ.tolist()
    none = torch.tensor([], dtype=torch.long, device=h1.device)
    e_phi = _active(h1, eri, occ, none.reshape(1, 0))[2][0]
    e_ref = torch.zeros((), dtype=torch.float64, device=h1.device)
    if ref:
        A = torch.tensor([ref], device=h1.device)
        e_ref = _lowest(h1, eri, occ, A, sum(occ_l[p] for p in ref))[0] - e_phi
    got, place = [], {}
    for n in orders:
        tuples = [t for t in itertools.combinations(exp, n)
                  if not skip or 0 < sum(occ_l[p] for p in (*ref, *t)) < len(ref) + n]
        if not tuples:
            got.append((tuples, None, None))
            continue
        A = torch.tensor([sorted((*ref, *t)) for t in tuples], device=h1.device)
        pairs = occ.long()[A].sum(1)
        eps = torch.zeros(len(tuples), dtype=torch.float64, device=h1.device)
        for k in sorted(set(pairs.tolist())):
            sel = (pairs == k).nonzero()[:, 0]
            low = torch.cat([_lowest(h1, eri, occ, part, k) for part in _chunks(A[sel], k)])
            # (one determinant: Phi itself)
            eps = eps.index_put((sel,), (0.0 * low if k in (0, A.shape[1]) else low - e_phi) - e_ref)
        inc = eps
        index = {t: i for i, t in enumerate(tuples)}
        for m in range(1, n):
            if not got[m - 1][0]:
                continue
            for sub in itertools.combinations(range(n), m):
                at = [place[m].get(tuple(t[i] for i in sub), -1) for t in tuples]
                at = torch.tensor(at, device=h1.device)
                inc = inc - torch.where(at >= 0, got[m - 1][2][at.clamp(min=0)], 0.0)
        place[n] = index
        got.append((tuples, eps, inc))
    total = e_phi + e_ref + sum(inc.sum() for _, _, inc in got if inc is not None)
    return got, e_phi, total


def _sigma(h1, eri, occ, cas, c):
    """H c of one active space: c -> E_rs c gathered for both spins, contracted, gathered back."""
    dev = h1.device
    A = torch.tensor([cas], device=dev)
    n, k = len(cas), int(sum(int(occ[p]) for p in cas))
    h, g, _ = _active(h1, eri, occ, A)
    ns = math.comb(n, k)
    C = c.reshape(ns, ns)
    lists = {pq: tuple(torch.tensor(v, device=dev, dtype=torch.long if i < 2 else torch.float64)
                       for i, v in enumerate(ijs)) for pq, ijs in _replacements(n, k).items()}
    hp = h[0] - 0.5 * torch.einsum("prrs->ps", g[0])
    out = torch.zeros_like(C)
    rows = max(1, 250_000_000 // (n * n * ns))
    # D[rs] = (E_rs (x) 1 + 1 (x) E_rs) C, in slabs of alpha strings
    D = torch.zeros((n * n, ns, ns), dtype=torch.float64, device=dev)
    for (r, s), (i, j, sg) in lists.items():
        if i.numel():
            D[r * n + s, i] += sg[:, None] * C[j]
            D[r * n + s][:, i] += sg[None, :] * C[:, j]
    G = g[0].reshape(n * n, n * n)
    for lo in range(0, ns, rows):
        part = D[:, lo:lo + rows]
        D[:, lo:lo + rows] = (0.5 * G @ part.reshape(n * n, -1) + hp.reshape(-1, 1) * C[lo:lo + rows].reshape(1, -1)
                              ).reshape(part.shape)
    for (p, q), (i, j, sg) in lists.items():
        if i.numel():
            out[i] += sg[:, None] * D[p * n + q, j]
            out[:, i] += sg[None, :] * D[p * n + q][:, j]
    return out.reshape(-1)


def exact(case, seed):
    dev = torch.device("cuda", 0)
    h1, eri, occ = (torch.tensor(x, device=dev) for x in _integrals(case, seed))
    task = case["task"]
    if task == "sigma":
        return _sigma(h1, eri, occ, _cas(case), _vector(case, occ.cpu().numpy(), seed))
    if task in ("solve", "type2"):
        return None
    ref, exp = _spaces(case, occ.cpu().numpy())
    orders = list(range(1, case["max_order"] + 1))
    # the orders whose dense diagonalisations take seconds (by the determinants of a tuple)
    counts = _tuple_counts(case)
    cost = {m: sum(c * (math.comb(len(ref) + m, k) ** 2) ** 2.5 for k, c in by_k.items()) for m, by_k in counts.items()}
    known = [m for m in orders if sum(cost[i] for i in range(1, m + 1)) <= 3.0e9 and sum(counts[m].values()) < 2e5]
    if task == "adjoint":
        if len(known) < len(orders):
            return None
        h1.requires_grad_(True)
        eri.requires_grad_(True)
        _, _, total = _expansion(h1, eri, occ, ref, exp, orders, case["skip"])
        total.backward()
        return dict(e_total=total.detach().reshape(1), grad_h1=h1.grad, grad_eri=eri.grad)
    got, e_phi, total = _expansion(h1, eri, occ, ref, exp, known, case["skip"])
    whole = len(known) == len(orders)
    n_out = len(orders)
    eps = [got[i][1] if i < len(known) else None for i in range(n_out)]
    inc = [got[i][2] if i < len(known) else None for i in range(n_out)]
    sums = torch.stack([h1.new_zeros(()) if x is None else x.sum() for x in inc]) if whole else None
    return dict(tuples=None, eps=eps, status=None, inc=inc, e_order=sums, e_phi=e_phi.reshape(1),
                e_total=total.reshape(1) if whole else None)
