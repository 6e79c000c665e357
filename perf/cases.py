"""Measured cases: the work that users of this library have it do, through its
public entry points, from the smallest sector contraction of a low-D sweep to
the 200-orbital CAS-SCF step.

A case is a dict of plain values.  Its "path" names the entry point:

* ``noalloc``     ``ops.hpsi_contract_noalloc``: one H_eff psi product on the
  caller's device buffers (torch tensors, torch's stream).
* ``contract``    ``ops.hpsi_contract``: the same product on host buffers.
* ``renormalize`` ``ops.grouped_gemm``: the two halves O U^T and U T of the
  renormalisation O' = U O U^T over all sector blocks of several operators.
* ``eigh``        ``ops.eigh_batched``: the density-matrix sectors of one
  decimation, or the two-orbital density matrices of the ordering step.
* ``transform``   ``ops.transform``: rotation of h and the Cholesky vectors.
* ``gradient``    ``ops.active_space`` and ``ops.orbital_gradient``.
* ``orbital_map`` ``autograd.orbital_transform``, forward and backward.
* ``job``         ``DMRG``: a float64 solve from the integrals to the RDMs.
* ``sweep``       ``DMRG.sweep`` of a split-precision context in mid-run.
* ``bond``        ``DMRG.bond_solve`` (split products, float64 check) there.

The sizes (sector dimensions, item counts, orbitals) follow from the case
alone, the numbers from the seed.  What the 3xTF32 products give carries about
22 significant bits, and a caller that asks for them keeps single precision:
those results are returned as float32.
"""
import math

import numpy as np
import torch

import paper_2503_20700_gb300 as pkg
import workloads
from paper_2503_20700_gb300 import autograd, ops

PREC = {"fp64": pkg.FP64, "split": pkg.SPLIT_TF32, "split-tc": pkg.SPLIT_HPSI_TC}


def listed():
    return [
        # the H_eff psi product of a low-D sweep (D of some tens: sectors of a
        # few multiplets), called in a loop by a program that owns the memory:
        # launches and latency
        dict(name="product small", path="noalloc", precision="fp64", sectors=14, lo=2, hi=24, ops=5),
        # a float64 product at D of about 512 (parity runs, Rayleigh quotients)
        dict(name="product f64", path="contract", precision="fp64", sectors=9, lo=40, hi=230, ops=6),
        # a split product with the sectors of a D = 2048 middle bond
        dict(name="product split", path="contract", precision="split-tc", sectors=5, lo=280, hi=600, ops=4),
        # renormalisation of a bond at D of about 1024 (ragged sectors)
        dict(name="renormalize", path="renormalize", sectors=11, lo=17, hi=410, ops=14),
        # spectra of the two-orbital density matrices of 30 orbitals
        dict(name="pair spectra", path="eigh", sectors=435, lo=16, hi=16),
        # the density-matrix sectors of a decimation at D of about 1024
        dict(name="decimation", path="eigh", sectors=13, lo=9, hi=601),
        # CAS-SCF on 200 orbitals, CAS(30,30), rank 600: the transformation, and
        # the active-space problem with the orbital gradient
        dict(name="transform", path="transform", nb=200, rank=600),
        dict(name="gradient", path="gradient", nb=200, rank=600, ncore=40, ncas=30),
        # a differentiable orbital rotation of a mid-sized molecule
        dict(name="orbital map", path="orbital_map", nb=75, rank=230, ncore=11, ncas=10),
        # naphthalene, 10 pi sites at D = 64: integrals to energy and RDMs
        dict(name="job naphthalene", path="job", rings=2, D=64, sweeps=2),
        # one more sweep of a split-precision run, and the solve of its middle
        # bond at a larger D
        dict(name="sweep split", path="sweep", n=16, rank=64, D=256),
        dict(name="bond split", path="bond", n=20, rank=80, D=512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["noalloc", "noalloc", "contract", "contract", "renormalize", "renormalize", "eigh", "eigh",
                       "transform", "transform", "gradient", "gradient", "orbital_map", "orbital_map", "job",
                       "sweep", "bond"])
    if path in ("noalloc", "contract"):
        hi = _log(rng, 9, 230)
        lo = max(1, int(hi * rng.uniform(0.1, 0.6)))
        c = dict(path=path, precision=rng.choice(["fp64", "split"]), sectors=rng.randint(3, 9), lo=lo, hi=hi,
                 ops=rng.randint(2, 6))
        if path == "contract" and rng.random() < 0.5:
            hi = _log(rng, 60, 600)
            c.update(precision="split-tc", lo=int(hi * rng.uniform(0.2, 0.6)), hi=hi, sectors=rng.randint(2, 5),
                     ops=rng.randint(2, 4))
        return c
    if path == "renormalize":
        hi = _log(rng, 12, 410)
        return dict(path=path, sectors=rng.randint(3, 11), lo=max(1, int(hi * rng.uniform(0.03, 0.5))), hi=hi,
                    ops=rng.randint(2, 14))
    if path == "eigh":
        hi = _log(rng, 12, 600)
        return dict(path=path, sectors=rng.randint(2, 13), lo=max(1, int(hi * rng.uniform(0.02, 0.5))), hi=hi)
    if path == "transform":
        nb = _log(rng, 12, 199)
        return dict(path=path, nb=nb, rank=int(nb * rng.uniform(1.5, 3.0)) + 1)
    if path == "gradient":
        nb = _log(rng, 14, 199)
        ncas = rng.randint(2, max(3, min(30, nb // 3)))
        return dict(path=path, nb=nb, rank=int(nb * rng.uniform(1.5, 3.0)) + 1,
                    ncore=rng.randint(0, (nb - ncas) // 2), ncas=ncas)
    if path == "orbital_map":
        nb = _log(rng, 8, 120)
        ncas = rng.randint(2, max(3, min(14, nb // 3)))
        return dict(path=path, nb=nb, rank=int(nb * rng.uniform(1.5, 3.0)) + 1,
                    ncore=rng.randint(0, (nb - ncas) // 2), ncas=ncas)
    if path == "job":
        return dict(path=path, rings=rng.choice([1, 2]), D=rng.randint(20, 63), sweeps=rng.randint(1, 2))
    n = rng.choice([12, 14, 15, 16])
    return dict(path=path, n=n, rank=rng.randint(3 * n, 4 * n), D=_log(rng, 70, 255))


# ------------------------------------------------------------------ structure
def _sector_dims(case, count):
    """Sector sizes of a block: the largest in the middle, Gaussian flanks."""
    x = np.linspace(-1.0, 1.0, count) if count > 1 else np.zeros(1)
    d = case["lo"] + (case["hi"] - case["lo"]) * np.exp(-4.0 * x * x)
    wob = np.random.default_rng([count, case["lo"], case["hi"]]).uniform(0.9, 1.0, count)
    return [max(1, case["lo"], int(v)) for v in d * wob]


def _product(case):
    """Blocks and items of one product: sigma block i gathers, for each of
    `ops` operator pairs, psi blocks i-1, i, i+1, with operators stored either
    way round, and the two identity terms (H_L, H_R)."""
    dl, dr = _sector_dims(case, case["sectors"]), _sector_dims(case, case["sectors"])[::-1]
    rng = np.random.default_rng([case["sectors"], case["lo"], case["hi"], case["ops"]])
    poff = np.concatenate([[0], np.cumsum([a * b for a, b in zip(dl, dr)])]).astype(int)
    alen = blen = 0
    blocks, items = [], []
    flops = 0.0
    for i, (m, n) in enumerate(zip(dl, dr)):
        first = len(items)
        terms = [(j, 0, 0) for _ in range(case["ops"]) for j in (i - 1, i, i + 1) if 0 <= j < len(dl)]
        for j, aid, bid in terms + [(i, 1, 0), (i, 0, 1)]:
            ka, kb = dl[j], dr[j]
            ta, tb = int(rng.integers(0, 2)), int(rng.integers(0, 2))
            items.append((0 if aid else alen, int(poff[j]), 0 if bid else blen, m if ta else ka, kb, n if tb else kb,
                          ta, tb, ka, kb, aid, bid, float(rng.uniform(-1.0, 1.0))))
            if not aid:
                alen += m * ka
                flops += 2.0 * m * ka * kb
            if not bid:
                blen += n * kb
                flops += 2.0 * m * n * kb
        blocks.append((int(poff[i]), m, n, n, first, len(items) - first))
    return blocks, items, alen, int(poff[-1]), blen, flops


def _renorm(case):
    """Groups and segments: T = O U^T (sector blocks O, d x d; U kept x d) and
    O' = U T (T given, d x kept), for `ops` operators on all sectors."""
    d = _sector_dims(case, case["sectors"])
    kept = [max(1, int(0.45 * x)) for x in d]
    uoff, u = [], 0
    for x, k in zip(d, kept):
        uoff.append(u)
        u += x * k
    groups, segs, a, c = [], [], 0, 0
    for _ in range(case["ops"]):
        for i, (x, k) in enumerate(zip(d, kept)):
            segs.append((a, uoff[i], x, x, x, 0, 1, 1.0))         # O (x x x) U^T
            groups.append((c, x, k, k, len(segs) - 1, 1))
            a += x * x
            c += x * k
    # U is read as the left operand here: it stands behind the O blocks in A,
    # and the T blocks behind the U blocks in B
    b = u
    for _ in range(case["ops"]):
        for i, (x, k) in enumerate(zip(d, kept)):
            segs.append((a + uoff[i], b, x, x, k, 0, 0, 1.0))     # U T
            groups.append((c, k, k, k, len(segs) - 1, 1))
            b += x * k
            c += k * k
    return d, kept, groups, segs, a, u, b, c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _host(t):
    return t.cpu().numpy()


def _orthogonal(g, n):
    return torch.linalg.qr(_normal(g, n, n))[0]


def _orbital_inputs(case, g):
    """h and Cholesky vectors that decay away from the diagonal (the random
    Cholesky form of ``workloads.cholesky_random``), made on the device."""
    nb, rank = case["nb"], case["rank"]
    h = _normal(g, nb, nb)
    h = 0.5 * (h + h.T) / math.sqrt(2.0) + torch.diag(torch.linspace(-2.0, -0.5, nb, device="cuda", dtype=torch.float64))
    p = torch.arange(nb, device="cuda", dtype=torch.float64)
    env = torch.exp(-(p[:, None] - p[None, :]).abs() / 6.0)
    x = _normal(g, rank, nb, nb)
    return h, math.sqrt(0.25 / rank) * env * (x + x.transpose(1, 2))


def _rdms(n, g):
    """RDM-shaped weights with the symmetries of a real wavefunction's."""
    x = _normal(g, n, n)
    gamma = torch.diag(torch.linspace(1.9, 0.1, n, device="cuda", dtype=torch.float64)) + 0.02 * (x + x.T)
    big = torch.einsum("ps,qr->pqrs", gamma, gamma) - 0.5 * torch.einsum("pr,qs->pqrs", gamma, gamma)
    y = 0.01 * _normal(g, n, n, n, n)
    y = y + y.permute(1, 0, 3, 2)
    return gamma, big + y + y.permute(3, 2, 1, 0)


def _context(case, seed):
    """A split-precision run on a random Cholesky active space, ramped to D:
    a sweep at 64 multiplets and one at D."""
    h, L = workloads.cholesky_random(case["n"], case["rank"], seed=int(seed))
    occ, path = workloads.aufbau_state(h, case["n"], 0)
    g = pkg.DMRG(h, chol=L, n_elec=case["n"], D=64, tol=1e-7, precision=pkg.SPLIT_HPSI_TC, max_iter=4, occ=occ,
                 two_s_right=path)
    g.sweep(1)
    g.set_bond_dim(case["D"])
    g.sweep(1)
    return g


def prepare(case, seed):
    pkg.load()
    path, g = case["path"], _gen(seed)
    s = {"path": path, "case": case}
    if path in ("noalloc", "contract"):
        s["blocks"], s["items"], na, npsi, nb, _ = _product(case)
        A, P, B = _normal(g, max(na, 1)), _normal(g, npsi), _normal(g, max(nb, 1))
        P /= P.norm()  # a two-site wavefunction
        if path == "noalloc":
            s.update(A=A, P=P, B=B, C=torch.zeros(npsi, device="cuda", dtype=torch.float64))
        else:
            s.update(A=_host(A), P=_host(P), B=_host(B))
    elif path == "renormalize":
        d, kept, s["groups"], s["segs"], na, nu, nb, s["clen"] = _renorm(case)
        U = torch.cat([_orthogonal(g, x)[:k].reshape(-1) for x, k in zip(d, kept)])
        s["A"] = _host(torch.cat([_normal(g, na), U]))
        s["B"] = _host(torch.cat([U, _normal(g, nb - nu)]))
    elif path == "eigh":
        s["mats"] = []
        for n in _sector_dims(case, case["sectors"]):
            q = _orthogonal(g, n)
            # weights over three decades: the eigenvectors of the (far smaller)
            # discarded ones are not determined to rounding
            u = torch.linspace(0.0, 1.0, n, device="cuda", dtype=torch.float64)
            w = 10.0 ** (-3.0 * u) * (1.0 + 0.2 / n * torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
            m = (q * (w / w.sum())) @ q.T
            s["mats"].append(_host(0.5 * (m + m.T)))
    elif path == "transform":
        h, L = _orbital_inputs(case, g)
        s.update(R=_host(_orthogonal(g, case["nb"])), h=_host(h), L=_host(L))
    elif path == "gradient":
        h, L = _orbital_inputs(case, g)
        gamma, Gamma = _rdms(case["ncas"], g)
        s.update(h=_host(h), L=_host(L), gamma=_host(gamma), Gamma=_host(Gamma))
    elif path == "orbital_map":
        h, L = _orbital_inputs(case, g)
        gamma, Gamma = _rdms(case["ncas"], g)
        kappa = 0.1 * _normal(g, case["nb"], case["nb"])
        s.update(h=h.cpu(), L=L.cpu(), kappa=kappa.cpu(), gh=gamma.cpu(),
                 ge=(0.5 * Gamma.permute(0, 3, 1, 2)).contiguous().cpu())
    elif path == "job":
        h, eri, ec = workloads.ppp_acene(case["rings"])
        # site energies of a substituted molecule (no spatial symmetry left)
        h = h + np.diag(0.03 * np.random.default_rng(int(seed)).standard_normal(len(h)))
        s.update(h=h, eri=eri, e_core=ec)
    elif path == "sweep":
        s["g"] = _context(case, seed)
    else:
        s["g"] = _context(case, seed)
        s["bond"] = case["n"] // 2 - 1
        s["g"].sweep_part(0, s["bond"] - 1)
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    path, case = s["path"], s["case"]
    if path == "noalloc":
        A, P, B, C = s["A"], s["P"], s["B"], s["C"]
        C.zero_()
        ops.hpsi_contract_noalloc(A.data_ptr(), A.numel(), P.data_ptr(), P.numel(), B.data_ptr(), B.numel(),
                                  C.data_ptr(), C.numel(), s["blocks"], s["items"], precision=PREC[case["precision"]],
                                  stream=torch.cuda.current_stream().cuda_stream)
        return C if case["precision"] == "fp64" else C.float()
    if path == "contract":
        C = np.zeros(s["P"].size)
        ops.hpsi_contract(s["A"], s["P"], s["B"], C, s["blocks"], s["items"], precision=PREC[case["precision"]])
        return C if case["precision"] == "fp64" else C.astype(np.float32)
    if path == "renormalize":
        return ops.grouped_gemm(s["A"], s["B"], np.zeros(s["clen"]), s["groups"], s["segs"])
    if path == "eigh":
        r = ops.eigh_batched(s["mats"])
        return {"w": np.concatenate([w for w, _ in r]), "v": np.concatenate([v.ravel() for _, v in r])}
    if path == "transform":
        return ops.transform(s["R"], s["h"], s["L"])
    if path == "gradient":
        e, ha, ea = ops.active_space(s["h"], s["L"], case["ncore"], case["ncas"])
        grad, fock = ops.orbital_gradient(s["h"], s["L"], case["ncore"], case["ncas"], s["gamma"], s["Gamma"],
                                          with_fock=True)
        return {"e": e, "h": ha, "eri": ea, "grad": grad, "fock": fock}
    if path == "orbital_map":
        kappa = s["kappa"].clone().requires_grad_(True)
        e, ha, ea = autograd.orbital_transform(kappa, s["h"], s["L"], case["ncore"], case["ncas"])
        torch.autograd.backward([e, ha, ea], [torch.ones_like(e), s["gh"], s["ge"]])
        return {"e": e.detach(), "h": ha.detach(), "eri": ea.detach(), "kappa": kappa.grad}
    if path == "job":
        g = pkg.DMRG(s["h"], eri=s["eri"], n_elec=len(s["h"]), D=case["D"], e_core=s["e_core"], tol=1e-12)
        e, _ = g.sweep(case["sweeps"])
        g1, g2 = g.rdm12()
        bonds = g.bond_energies()
        g.close()
        return {"e": e, "bonds": bonds, "rdm1": g1, "rdm2": g2}
    if path == "sweep":
        e, _ = s["g"].sweep(1)
        return {"e": np.float32(e)}
    r = s["g"].bond_solve(s["bond"], 0, pkg.SPLIT_HPSI_TC, max_iter=12, tol=1e-7, min_calls=12)
    return {"e": np.float32(r["energy"]), "rq": np.float32(r["energy_rq64"]), "dim": int(r["dim"])}


# ------------------------------------------------------------------ work
def work(case):
    path = case["path"]
    if path in ("noalloc", "contract"):
        _, _, na, npsi, nb, flops = _product(case)
        return {"bytes": 8.0 * (na + nb + 2 * npsi), "flops": flops}
    if path == "renormalize":
        d, kept, _, _, na, nu, nb, nc = _renorm(case)
        return {"bytes": 8.0 * (na + nb + nc),
                "flops": case["ops"] * sum(2.0 * x * x * k + 2.0 * k * k * x for x, k in zip(d, kept))}
    if path == "eigh":
        d = _sector_dims(case, case["sectors"])
        # tridiagonalisation, and the eigenvectors carried back
        return {"bytes": 16.0 * sum(n * n for n in d), "flops": sum(4.0 / 3 * n**3 + 2.0 * n**3 for n in d)}
    if path in ("transform", "gradient", "orbital_map"):
        nb, rank = case["nb"], case["rank"]
        rot = 4.0 * nb**3 * (rank + 1)
        if path == "transform":
            return {"bytes": 8.0 * (2 * (rank + 1) + 1) * nb * nb, "flops": rot}
        nc, na = case["ncore"], case["ncas"]
        core = 2.0 * rank * nb * nb * (1 + nc)          # J and K of the core
        eri = 2.0 * rank * na**4
        fock = core + 2.0 * rank * nb * nb * (1 + na) + 2.0 * rank * nb * na * na + eri + 2.0 * rank * nb * na * na
        vals = (rank + 2) * nb * nb + na**4
        if path == "gradient":
            return {"bytes": 8.0 * (vals + 2 * na**4), "flops": core + eri + fock}
        # exponential and its adjoint by one Pade-like sequence of products each
        return {"bytes": 8.0 * (2 * vals + 2 * na**4), "flops": rot + core + eri + fock + 24.0 * nb**3}
    # whole runs: two-site Davidson steps of sector blocks; the floating-point
    # work of the products, with the sector structure taken as one dense block
    # per 12 sectors, and the operators of a bond read once per product
    if path == "job":
        n, D, steps = 4 * case["rings"] + 2, case["D"], 2 * case["sweeps"] * 8
    elif path == "sweep":
        n, D, steps = case["n"], case["D"], 4 * 2 * (case["n"] - 2)
    else:
        n, D, steps = case["n"], case["D"], 13
    D = min(D, 4 ** (n // 2) / (n / 2.0 + 1))
    pairs = n * n / 2.0
    return {"bytes": 8.0 * pairs * D * D / 6.0 * steps / 4.0, "flops": 4.0 * pairs * 3.0 * D**3 / 12.0 * steps}


# ------------------------------------------------------------------ 64 bits
def _exact_product(case, s):
    A, P, B = (torch.as_tensor(s[k]).cuda() for k in "APB")
    C = torch.zeros(P.numel(), device="cuda", dtype=torch.float64)
    for c0, m, n, _, i0, cnt in s["blocks"]:
        out = C[c0:c0 + m * n].view(m, n)
        for a, p, b, _, _, _, ta, tb, ka, kb, aid, bid, al in s["items"][i0:i0 + cnt]:
            x = al * P[p:p + ka * kb].view(ka, kb)
            if not aid:
                x = (A[a:a + m * ka].view(ka, m).T if ta else A[a:a + m * ka].view(m, ka)) @ x
            if not bid:
                x = x @ (B[b:b + n * kb].view(kb, n) if tb else B[b:b + n * kb].view(n, kb).T)
            out += x
    return C


def _exact_fock(h, L, nc, na, gamma, Gamma):
    """Core energy, inactive Fock matrix, active integrals and (with RDMs)
    the generalised Fock matrix of a closed-shell core and an active space."""
    a = slice(nc, nc + na)
    v = torch.einsum("kii->k", L[:, :nc, :nc])
    FI = h + 2.0 * torch.einsum("k,kpq->pq", v, L) - torch.einsum("kpi,kiq->pq", L[:, :, :nc], L[:, :nc, :])
    e = torch.diagonal(h)[:nc].sum() + torch.diagonal(FI)[:nc].sum()
    La = L[:, a, a]
    eri = torch.einsum("ktu,kvw->tuvw", La, La)
    if gamma is None:
        return e, FI[a, a], eri, None
    FA = torch.einsum("k,kpq->pq", torch.einsum("tu,ktu->k", gamma, La), L)
    FA = FA - 0.5 * torch.einsum("kpu,kuq->pq", L[:, :, a] @ gamma, L[:, a, :])
    W = torch.einsum("tvwu,kvw->ktu", Gamma, La)
    F = torch.zeros_like(h)
    F[:nc] = 2.0 * (FI + FA).T[:nc]
    F[a] = gamma @ FI[:, a].T + torch.einsum("ktu,kqu->tq", W, L[:, :, a])
    return e, FI[a, a], eri, F


def exact(case, seed):
    path = case["path"]
    if path in ("job", "sweep", "bond"):
        return None
    s = prepare(case, seed)
    if path in ("noalloc", "contract"):
        return _exact_product(case, s)
    if path == "renormalize":
        A, B = torch.as_tensor(s["A"]).cuda(), torch.as_tensor(s["B"]).cuda()
        C = torch.zeros(s["clen"], device="cuda", dtype=torch.float64)
        for c0, m, n, _, i0, _ in s["groups"]:
            a, b, k, _, _, _, tb, _ = s["segs"][i0]
            y = B[b:b + n * k].view(n, k).T if tb else B[b:b + n * k].view(k, n)
            C[c0:c0 + m * n] = (A[a:a + m * k].view(m, k) @ y).reshape(-1)
        return C
    if path == "eigh":
        ws, vs = [], []
        for m in s["mats"]:
            w, v = np.linalg.eigh(m)
            w, v = w[::-1], v[:, ::-1].T
            v = v * np.sign(v[np.arange(len(w)), np.argmax(np.abs(v), axis=1)])[:, None]
            ws.append(w)
            vs.append(v.ravel())
        return {"w": np.concatenate(ws), "v": np.concatenate(vs)}
    if path == "transform":
        R, h, L = (torch.as_tensor(s[k]).cuda() for k in ("R", "h", "L"))
        return R.T @ h @ R, R.T @ L @ R
    if path == "gradient":
        h, L, gamma, Gamma = (torch.as_tensor(s[k]).cuda() for k in ("h", "L", "gamma", "Gamma"))
        e, ha, eri, F = _exact_fock(h, L, case["ncore"], case["ncas"], gamma, Gamma)
        grad = 2.0 * (F - F.T)
        a = slice(case["ncore"], case["ncore"] + case["ncas"])
        grad[a, a] = 0.0
        return {"e": float(e), "h": ha, "eri": eri, "grad": grad, "fock": F}
    h, L, gh, ge = (s[k].cuda() for k in ("h", "L", "gh", "ge"))
    kappa = s["kappa"].cuda().requires_grad_(True)
    K = torch.tril(kappa, -1)
    R = torch.linalg.matrix_exp(K.T - K)
    e, ha, eri, _ = _exact_fock(R.T @ h @ R, R.T @ L @ R, case["ncore"], case["ncas"], None, None)
    torch.autograd.backward([e, ha, eri], [torch.ones_like(e), gh, ge])
    return {"e": e.detach(), "h": ha.detach(), "eri": eri.detach(), "kappa": kappa.grad}
