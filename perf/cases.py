"""The work that users of this library have it do, as cases to be timed and compared.

A case is one of four kinds:

``build``     one energy + Lagrangian build and its adjoint at a prepared B (the inner call of
              every orbital iteration), through the autograd function, the Builder, or the call
              on host buffers; optionally with the integrals J, K and the NOF-MP2 energies.
``geometry``  a new molecular geometry: B converted, then one build and its adjoint.
``scan``      many uneven instances (a dissociation scan) as one CUDA-graph replay.
``orbitals``  the hand-off to the orbital update: the Fockian, its double eigendecomposition,
              the rotated and reorthonormalised orbitals.

Inputs follow the recipe of the repository's synthetic workloads: slices of B symmetric, their
elements N(0, 1/2) exp(-|mu - nu| / 4) / sqrt(naux); h with a diagonal of -U(1, 10); orthonormal
C; strong gammas U(0, 1.45), the hole of each pair split by Dirichlet(1).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2004_06142_gb300 as dn

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # the smallest call: five pairs in a minimal basis; launches and latency are all of it
        dict(name="plain_fp64", kind="build", entry="autograd", nbf=24, naux=96, npair=5, ncwo=1,
             nsingle=0, functional=7, packed=False, mixed=False, blocks=1, integrals=False),
        dict(name="plain_mixed", kind="build", entry="builder", nbf=24, naux=96, npair=5, ncwo=1,
             nsingle=0, functional=7, packed=False, mixed=True, blocks=1, integrals=False),
        # a small open-shell molecule with the other functional, odd sizes, packed B, the
        # integrals and the NOF-MP2 energies of a final evaluation
        dict(name="multiplet_fp64", kind="build", entry="builder", nbf=97, naux=331, npair=4,
             ncwo=3, nsingle=3, functional=8, packed=True, mixed=False, blocks=1, integrals=True),
        # a small molecule in a double-zeta basis, differentiated: training-style use of the
        # energy as an autograd function, in double and in mixed precision
        dict(name="differentiation_fp64", kind="build", entry="autograd", nbf=120, naux=480,
             npair=8, ncwo=4, nsingle=0, functional=7, packed=False, mixed=False, blocks=1,
             integrals=False),
        dict(name="differentiation_mixed", kind="build", entry="autograd", nbf=120, naux=480,
             npair=8, ncwo=4, nsingle=0, functional=7, packed=False, mixed=True, blocks=1,
             integrals=False),
        # the medium molecule: the double path that final energies and error checks are taken
        # with, and the mixed path called from a driver whose orbitals live on the host
        dict(name="precision_fp64", kind="build", entry="builder", nbf=500, naux=2000, npair=20,
             ncwo=3, nsingle=0, functional=7, packed=False, mixed=False, blocks=1,
             integrals=False),
        dict(name="precision_mixed_host", kind="build", entry="host", nbf=500, naux=2000,
             npair=20, ncwo=3, nsingle=0, functional=7, packed=False, mixed=True, blocks=1,
             integrals=False),
        # the largest molecule, packed B: one orbital iteration's build and adjoint
        dict(name="large_mixed", kind="build", entry="builder", nbf=1200, naux=4800, npair=50,
             ncwo=2, nsingle=0, functional=7, packed=True, mixed=True, blocks=1,
             integrals=False),
        # one more geometry of a ragged medium molecule: new integrals, converted and built once
        dict(name="new_geometry", kind="geometry", entry="builder", nbf=301, naux=1103, npair=10,
             ncwo=3, nsingle=0, functional=7, packed=True, mixed=True, blocks=1,
             integrals=False),
        # a dissociation scan of 64 uneven geometries, replayed
        dict(name="scan_64", kind="scan", count=64, nbf_min=40, nbf_max=240, npair=5),
        # the diagonalisation step of the orbital optimisation, of a small and of the largest
        # molecule
        dict(name="orbitals_small", kind="orbitals", nbf=120, nact=40),
        dict(name="orbitals_large", kind="orbitals", nbf=1200, nact=150),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "build", "geometry", "scan", "orbitals"])
    if kind == "orbitals":
        n = _log_int(rng, 24, 1200)
        return dict(kind=kind, nbf=n, nact=rng.randint(max(1, n // 10), max(1, n // 2)))
    if kind == "scan":
        lo = _log_int(rng, 24, 120)
        return dict(kind=kind, count=_log_int(rng, 4, 64), nbf_min=lo,
                    nbf_max=rng.randint(lo, 240), npair=rng.randint(2, 6))
    mixed = rng.random() < 0.5 if kind == "build" else True
    while True:
        nbf = _log_int(rng, 24, 1200 if mixed else 500)
        naux = int(nbf * rng.uniform(2.0, 4.5))
        nact = rng.randint(max(4, nbf // 16), max(4, min(nbf // 2, 250)))
        ncwo = rng.randint(1, 4)
        npair = max(1, nact // (1 + ncwo))
        nsingle = rng.choice([0, 0, 1, 3])
        nact = npair * (1 + ncwo) + nsingle
        flops = 2.0 * naux * nbf * nact * (nbf + 2 * nact)
        # no more than the listed medium (double) or large (mixed) case
        if nact <= min(nbf, 250) and flops <= (2.6e12 if mixed else 1.05e11):
            break
    entry = rng.choice(["autograd", "builder", "host"]) if kind == "build" else "builder"
    return dict(kind=kind, entry=entry, nbf=nbf, naux=naux, npair=npair, ncwo=ncwo,
                nsingle=nsingle, functional=rng.choice([5, 7, 7, 8]),
                packed=rng.random() < 0.5, mixed=mixed, blocks=rng.choice([1, 1, 1, 3]),
                integrals=entry == "builder" and rng.random() < 0.3)


# ---------------------------------------------------------------------------- inputs
def _gen(seed, tag):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + tag) % (1 << 62))
    return g


def _B_block(nbf, naux, packed, seed, p0, p1):
    """Slices p0..p1 (one stream per block of slices)."""
    g = _gen(seed, 16 + p0)
    i = torch.arange(nbf, device=DEV)
    band = torch.exp(-(i[:, None] - i[None, :]).abs().to(F64) / 4.0) / math.sqrt(naux)
    # an off-diagonal element is the mean of two N(0, 1) draws, a diagonal one is N(0, 1)
    band = band * torch.where(i[:, None] == i[None, :], 1.0, math.sqrt(0.5)).to(F64)
    mu, nu = torch.tril_indices(nbf, nbf, device=DEV)
    tri = torch.randn(p1 - p0, mu.numel(), dtype=F64, device=DEV, generator=g)
    tri.mul_(band[mu, nu])
    if packed:
        return tri
    out = torch.empty(p1 - p0, nbf, nbf, dtype=F64, device=DEV)
    out[:, mu, nu] = tri
    out[:, nu, mu] = tri
    return out


def _blocks_of(nbf, naux):
    step = max(1, min(naux, int(3e8 // (nbf * nbf))))
    return [(p, min(naux, p + step)) for p in range(0, naux, step)]


def _B(nbf, naux, packed, seed):
    shape = (naux, nbf * (nbf + 1) // 2) if packed else (naux, nbf, nbf)
    B = torch.empty(shape, dtype=F64, device=DEV)
    for p0, p1 in _blocks_of(nbf, naux):
        B[p0:p1] = _B_block(nbf, naux, packed, seed, p0, p1)
    return B


def _orthonormal(nbf, rng):
    return np.ascontiguousarray(np.linalg.qr(rng.standard_normal((nbf, nbf)))[0])


def _small_inputs(c, seed):
    """h, C, gamma, pair_map as numpy arrays."""
    nbf, npair, ncwo, ns = c["nbf"], c["npair"], c["ncwo"], c["nsingle"]
    rng = np.random.default_rng([int(seed), 1])
    i = np.arange(nbf)
    h = np.triu(rng.normal(0.0, 0.1, (nbf, nbf)) * np.exp(-np.abs(i[:, None] - i) / 4.0), 1)
    h = h + h.T
    h[i, i] = -rng.uniform(1.0, 10.0, nbf)
    C = _orthonormal(nbf, rng)
    gs = rng.uniform(0.0, 1.45, npair)
    weak = np.zeros((npair, ncwo - 1))
    for g in range(npair):
        hole = rest = 0.5 * math.sin(gs[g]) ** 2
        for k, part in enumerate(rng.dirichlet(np.ones(ncwo))[:-1] * hole):
            weak[g, k] = math.asin(math.sqrt(min(1.0, max(0.0, part / rest)))) if rest > 0 else 0.0
            rest *= math.cos(weak[g, k]) ** 2
    gamma = np.concatenate([gs, weak.reshape(-1)])
    pm = np.concatenate([np.arange(npair + ns), np.repeat(np.arange(npair), ncwo)])
    return h, C, gamma, pm.astype(np.int32)


def _nact(c):
    return c["npair"] * (1 + c["ncwo"]) + c["nsingle"]


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _scan_instances(c, seed):
    out = []
    for i in range(c["count"]):
        rng = np.random.default_rng([i, 4])  # the sizes of a scan are the molecule's, not the seed's
        nbf = int(rng.integers(c["nbf_min"], c["nbf_max"] + 1))
        ncwo = min(int(rng.integers(1, 5)), nbf // c["npair"] - 1)
        out.append(dict(nbf=nbf, naux=4 * nbf, npair=c["npair"], ncwo=ncwo, nsingle=0,
                        functional=7, packed=False))
    return out, [int(seed) * 64 + i for i in range(c["count"])]


def _orbital_inputs(c, seed):
    """A Lagrangian some iterations into an optimisation (its asymmetry small next to the
    spread of the diagonal, zero columns for the empty orbitals), the previous eigenvalues in
    decreasing order, and the orbitals."""
    n, a = c["nbf"], c["nact"]
    rng = np.random.default_rng([int(seed), 2])
    lam = np.zeros((n, n))
    lam[:, :a] = rng.normal(0.0, 0.05, (n, a))
    lam[:a, :a] += -np.diag(rng.uniform(0.1, 10.0, a))
    fdiag = np.sort(rng.uniform(-10.0, 10.0, n))[::-1]
    return lam, np.ascontiguousarray(fdiag), _orthonormal(n, rng)


# ---------------------------------------------------------------------------- the calls
def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "orbitals":
        lam, fdiag, C = _orbital_inputs(c, seed)
        s = dict(c=c, lam=_dev(lam), fdiag=_dev(fdiag), C=_dev(C))
        s["C_new"], s["eps"] = torch.empty_like(s["C"]), torch.empty_like(s["fdiag"])
        s["ws"] = dn.donof_orbital_update(s["lam"], s["fdiag"], s["C"], s["C_new"], s["eps"])
        return s
    if c["kind"] == "scan":
        insts, seeds = _scan_instances(c, seed)
        sizes = dict(E=1, lam=0, dE_dgamma=0, dE_dC=0)
        offs = []
        for x in insts:
            o = {}
            for k, n in (("E", 1), ("lam", x["nbf"] ** 2), ("dE_dgamma", x["npair"] * x["ncwo"]),
                         ("dE_dC", x["nbf"] ** 2)):
                if k == "E":
                    o[k] = (len(offs), 1)
                else:
                    o[k] = (sizes[k], n)
                    sizes[k] += n
            offs.append(o)
        sizes["E"] = len(insts)
        # one buffer per output, an instance's part behind the one before it
        out = {k: torch.zeros(n, dtype=F64, device=DEV) for k, n in sizes.items()}
        probs, rows = [], []
        for x, o, sd in zip(insts, offs, seeds):
            h, C, gamma, pm = _small_inputs(x, sd)
            probs.append(dn.make_problem(x["nbf"], x["naux"], x["npair"], x["ncwo"], dn.PNOF7,
                                         dn.B_DENSE, dn.MIXED))
            row = dict(h=_dev(h), B=_B(x["nbf"], x["naux"], False, sd), C=_dev(C),
                       gamma=_dev(gamma), pair_map=_dev(pm))
            for k, (at, n) in o.items():
                row[k] = out[k][at:at + n]
            rows.append(row)
        batch = dn.Batch(probs, rows)
        batch.prepare()
        batch.run(0)  # the energies of the scan first, then a first pass with gradients
        batch.run(dn.BATCH_BACKWARD)
        return dict(c=c, batch=batch, out=out)
    h, C, gamma, pm = _small_inputs(c, seed)
    s = dict(c=c, h=_dev(h), pm=_dev(pm), B=_B(c["nbf"], c["naux"], c["packed"], seed),
             one=torch.ones(1, dtype=F64, device=DEV))
    budget = 0
    if c["blocks"] > 1:  # a driver short of memory: the auxiliary index streamed in blocks
        budget = c["naux"] * c["nbf"] * _nact(c) * 24 // c["blocks"]
    s["bld"] = dn.Builder(c["nbf"], c["naux"], c["npair"], c["ncwo"], c["functional"],
                          dn.B_PACKED if c["packed"] else dn.B_DENSE,
                          dn.MIXED if c["mixed"] else dn.FP64, x_budget_bytes=budget,
                          nsingle=c["nsingle"])
    if c["kind"] == "build":
        s["bld"].prepare(s["B"])
    if c["entry"] == "host":
        pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()  # noqa: E731
        n, ng = c["nbf"], c["npair"] * c["ncwo"]
        s["C"], s["gamma"] = pin(C), pin(gamma)
        s["E"], s["lam"], s["dg"], s["dC"] = (
            torch.zeros(shape, dtype=F64).pin_memory() for shape in ((1,), (n, n), (ng,), (n, n)))
        s["staging"] = dn.alloc_workspace(dn.donof_host_staging_size(s["bld"].prob), DEV)
    else:
        s["C"], s["gamma"] = _dev(C), _dev(gamma)
        if c["entry"] == "autograd":
            s["C"].requires_grad_(True)
            s["gamma"].requires_grad_(True)
    return s


def run(state):
    s, c = state, state["c"]
    if c["kind"] == "orbitals":
        dn.donof_orbital_update(s["lam"], s["fdiag"], s["C"], s["C_new"], s["eps"], s["ws"])
        return dict(C_new=s["C_new"], eps=s["eps"])
    if c["kind"] == "scan":
        s["batch"].run(dn.BATCH_BACKWARD | dn.BATCH_GRAPH)
        return s["out"]
    bld = s["bld"]
    if c["kind"] == "geometry":
        bld.prepare(s["B"])
    if c["entry"] == "host":
        dn.donof_energy_lagrangian_host(bld.prob, s["h"], s["B"], s["C"], s["gamma"], s["pm"],
                                        bld.ws, s["staging"], s["E"], s["lam"], s["dg"], s["dC"])
        return dict(E=s["E"], lam=s["lam"], dE_dgamma=s["dg"], dE_dC=s["dC"])
    if c["entry"] == "autograd":
        E, lam = dn.energy(s["C"], s["gamma"], bld, s["h"], s["pm"])
        dC, dg = torch.autograd.grad(E, (s["C"], s["gamma"]))
        return dict(E=E.detach(), lam=lam, dE_dgamma=dg, dE_dC=dC)
    E, lam, dg = bld.forward(s["h"], s["C"], s["gamma"], s["pm"])
    dC, _ = bld.backward(s["one"])
    out = dict(E=E, lam=lam, dE_dgamma=dg, dE_dC=dC)
    if c["integrals"]:
        out["J"], out["K"] = bld.jk()
        out["E_hf"], out["E_sta"] = bld.nofmp2_static(s["pm"])
    return out


# ---------------------------------------------------------------------------- what a pass needs
def _build_work(c, b_bytes):
    n, q, a = c["nbf"], c["naux"], _nact(c)
    tri = q * (n * (n + 1) // 2)
    return (tri * b_bytes + 8 * (4 * n * n),  # B, h, C in; lambda, dE/dC out
            2.0 * q * n * a * (n + 2 * a) + 4.0 * n * n * a)


def work(case):
    c = case
    if c["kind"] == "orbitals":
        n = c["nbf"]
        # reduction to tridiagonal form, eigenvectors taken back, C V, reorthonormalisation
        return dict(bytes=8.0 * 3 * n * n, flops=(4.0 / 3 + 2 + 2 + 4) * n ** 3)
    if c["kind"] == "scan":
        parts = [_build_work(x, 4) for x in _scan_instances(c, 0)[0]]
        return dict(bytes=float(sum(p[0] for p in parts)), flops=float(sum(p[1] for p in parts)))
    # a mixed build reads the converted B (two half-precision planes), a double one B itself,
    # and a new geometry B itself besides
    byts, flops = _build_work(c, 4 if c["mixed"] else 8)
    if c["kind"] == "geometry":
        byts += 2 * 4 * c["naux"] * (c["nbf"] * (c["nbf"] + 1) // 2)
    return dict(bytes=float(byts), flops=float(flops))


# ---------------------------------------------------------------------------- in 64 bits
def _occupations(gamma, c):
    """n, sqrt(n), Phi over the active orbitals, differentiable in gamma."""
    npair, ncwo, ns = c["npair"], c["ncwo"], c["nsingle"]
    gs, gw = gamma[:npair], gamma[npair:].reshape(npair, ncwo - 1)
    one = torch.ones(npair, 1, dtype=F64, device=gamma.device)
    hole = gs.sin().abs() / math.sqrt(2.0)
    before = torch.cumprod(torch.cat([one, gw.cos().abs()], 1), 1)
    sq_w = hole[:, None] * before * torch.cat([gw.sin().abs(), one], 1)
    n_s = 0.5 * (1.0 + gs.cos() ** 2)
    half = torch.full((ns,), 0.5, dtype=F64, device=gamma.device)
    n = torch.cat([n_s, half, (sq_w ** 2).reshape(-1)])
    sq = torch.cat([n_s.sqrt(), half.sqrt(), sq_w.reshape(-1)])
    hole_of = torch.cat([hole, half.sqrt(), (1.0 - sq_w ** 2).sqrt().reshape(-1)])
    return n, sq, sq * hole_of


def _energies(H, J, K, gamma, pm, c):
    """E, and the reference and static energies of NOF-MP2."""
    npair, ns = c["npair"], c["nsingle"]
    n, sq, phi = _occupations(gamma, c)
    a = n.numel()
    idx = torch.arange(a, device=H.device)
    same = pm[:, None] == pm[None, :]
    single = (idx >= npair) & (idx < npair + ns)
    strong = idx < npair
    sign = torch.where((idx[:, None] != idx[None, :]) & (strong[:, None] ^ strong[None, :]), -1.0, 1.0)
    pi = torch.where(same & ~single[:, None], sign * sq[:, None] * sq[None, :], 0.0)
    other = (~same).to(F64)
    nn, pp = n[:, None] * n[None, :], phi[:, None] * phi[None, :]
    E = 2.0 * (n * H).sum() + (pi * K).sum() + (other * nn * (2.0 * J - K)).sum()
    if c["functional"] == 7:
        E = E - (other * pp * K).sum()
    elif c["functional"] == 8:
        E = E - (other * 4.0 * pp ** 2 * K).sum()
    w = torch.where(single, 0.5, torch.where(strong, 1.0, 0.0)).to(F64)
    e_hf = 2.0 * (w * H).sum() + (w[:, None] * w[None, :] * (2.0 * J - K)).sum()
    e_hf = e_hf - (single * J.diagonal()).sum() / 4.0
    lam = 1.0 - (1.0 - 2.0 * n).abs()
    off = (idx[:, None] != idx[None, :]).to(F64)
    e_sta = (off * (lam[:, None] * lam[None, :]).clamp(min=0).sqrt() * pi * K).sum()
    return E, e_hf, e_sta - 4.0 * (other * pp ** 2 * K).sum()


def _exact_build(c, seed):
    n, a = c["nbf"], _nact(c)
    h, C, gamma, pm = (_dev(x) for x in _small_inputs(c, seed))
    pm = pm.long()
    Ca = C[:, :a].contiguous()
    mu, nu = torch.tril_indices(n, n, device=DEV)

    def slices(p0, p1):
        tri = _B_block(n, c["naux"], c["packed"], seed, p0, p1)
        if not c["packed"]:
            return tri
        out = torch.empty(p1 - p0, n, n, dtype=F64, device=DEV)
        out[:, mu, nu] = tri
        out[:, nu, mu] = tri
        return out

    J = torch.zeros(a, a, dtype=F64, device=DEV)
    K = torch.zeros_like(J)
    kept = []
    for p0, p1 in _blocks_of(n, c["naux"]):
        X = (slices(p0, p1).reshape(-1, n) @ Ca).reshape(p1 - p0, n, a)
        b = Ca.T @ X
        d = b.diagonal(dim1=1, dim2=2)
        J += d.T @ d
        K += (b * b).sum(0)
        kept.append((X, b))
    H = ((h @ Ca) * Ca).sum(0)
    leaf = [t.detach().clone().requires_grad_(True) for t in (H, J, K, gamma)]
    E, e_hf, e_sta = _energies(*leaf, pm, c)
    gH, gJ, gK, dg = torch.autograd.grad(E, leaf)
    gJ, gK = gJ + gJ.T, gK + gK.T
    dC = torch.zeros(n, n, dtype=F64, device=DEV)
    dC[:, :a] = 2.0 * (h @ Ca) * gH
    for X, b in kept:
        gb = b * gK
        d = b.diagonal(dim1=1, dim2=2)
        gb.diagonal(dim1=1, dim2=2).add_(d @ gJ)
        # E depends on b = Ca^T B Ca: dE/dCa = 2 X gb (B and gb symmetric)
        dC[:, :a] += 2.0 * torch.bmm(X, gb).sum(0) if X.shape[0] < 8 else 2.0 * (
            X.permute(1, 0, 2).reshape(n, -1) @ gb.reshape(-1, a))
    out = dict(E=E.detach(), lam=C.T @ dC / 4.0, dE_dgamma=dg, dE_dC=dC)
    if c["entry"] != "autograd":
        out["E"] = out["E"].reshape(1)
    if c["integrals"]:
        out.update(J=J, K=K, E_hf=e_hf.detach().reshape(1), E_sta=e_sta.detach().reshape(1))
    return out


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "orbitals":
        lam, fdiag, _ = _orbital_inputs(c, seed)
        F = np.triu(lam - lam.T, 1)
        F = F + F.T + np.diag(fdiag)
        # eigenvectors are defined up to sign only
        return dict(C_new=None, eps=torch.from_numpy(np.linalg.eigvalsh(F)))
    if c["kind"] == "scan":
        outs = [_exact_build(dict(x, entry="builder", integrals=False), sd)
                for x, sd in zip(*_scan_instances(c, seed))]
        return {k: torch.cat([o[k].reshape(-1) for o in outs])
                for k in ("E", "lam", "dE_dgamma", "dE_dC")}
    return _exact_build(c, seed)
