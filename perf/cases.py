"""The performance cases of the DSRG-MRPT2 library: what its users have it do,
through the public entry points of ``paper_1603_00561_gb300``, over the real
range of molecule sizes.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes a case's inputs on the GPU from a seed together with the plan
that a program keeps, ``run`` is one pass, ``work`` the bytes and operations of
a pass that the path cannot do without, and ``exact`` the same outputs from
plain torch in FP64.

Inputs follow the distributions of the repository's synthetic molecules: DF
factors b N(0,1) e^{-0.02 Q}, orbital energies core U[-2, -0.3], active
U[-0.2, 0.1], virtual U[0.05, 5], a density with eigenvalues in [0, 2] and
trace nA, small cumulants.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1603_00561_gb300 as pk

F8 = torch.float64


def _case(name, kind, nC, nA, nV, naux, precision="bf16x3", s=0.5, ext=False):
    return {"name": name, "kind": kind, "ncore": nC, "nactive": nA, "nvirt": nV, "naux": naux,
            "precision": precision, "s": s, "ext": ext}


def listed():
    return [
        # a small system (74 orbitals): one call of a scan or a test, all launches
        _case("tiny-energy-bf16x3", "energy", 10, 4, 60, 200),
        # the same system in the default FP64 plan, with the gradient that a
        # geometry step or a finite-difference check asks for
        _case("tiny-gradient-fp64", "gradient", 10, 4, 60, 200, "fp64"),
        # (2,3)-naphthyne in cc-pVTZ: the everyday energy
        _case("vtz-energy-bf16x3", "energy", 24, 2, 372, 1200),
        # the same molecule in the default FP64 plan: the reference energies
        _case("vtz-energy-fp64", "energy", 24, 2, 372, 1200, "fp64"),
        # its gradient with the split plan
        _case("vtz-gradient-bf16x3", "gradient", 24, 2, 372, 1200),
        # (2,3)-naphthyne in cc-pV5Z, the largest molecule: inputs on the device
        _case("v5z-energy-bf16x3", "energy", 24, 2, 1214, 3400),
        # ... and through the host-buffer call, from pinned memory
        _case("v5z-host-bf16x3", "host", 24, 2, 1214, 3400),
        # odd sizes, a larger active space, TF32x3, three-body cumulant and
        # off-diagonal Fock block: the full Table 1
        _case("odd-full-table1-tf32x3", "energy", 31, 5, 467, 1609, "tf32x3", 1.0, True),
        # a batch of uneven molecules (nC 8-40, nA 2-6, nV 100-600), one graph
        {"name": "batch16-bf16x3", "kind": "batch", "molecules": 16, "sizes_seed": 0,
         "precision": "bf16x3", "s": 0.5},
        # Fock matrix and semicanonical orbitals of the cc-pVTZ molecule
        _case("vtz-semicanonical", "semicanonical", 24, 2, 372, 1200, "fp64"),
        # its DF factors (holes x particles) from AO three-centre integrals
        _case("vtz-df-transform", "df", 24, 2, 372, 1200, "fp64"),
        # Cholesky vectors of a small basis from 240 factors at the usual 1e-5
        {"name": "cholesky-n56", "kind": "cholesky", "nbf": 56, "nfac": 240, "tau": 1e-5},
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], uniform in its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _pair_work(nC, nV, naux):
    return nC * (nC + 1) * naux * nV * nV


def draw(rng):
    kind = rng.choices(["energy", "gradient", "host", "batch", "semicanonical", "df", "cholesky"],
                       [8, 4, 2, 2, 2, 2, 1])[0]
    if kind == "batch":
        return {"kind": kind, "molecules": _log(rng, 3, 16), "sizes_seed": rng.randrange(1, 1 << 20),
                "precision": rng.choice(["bf16x3", "bf16x3", "tf32x3"]), "s": rng.choice([0.1, 0.5, 1.0])}
    if kind == "cholesky":
        n = _log(rng, 10, 56)
        # thresholds below the last factor, so that the rank is the number of factors
        return {"kind": kind, "nbf": n, "nfac": min(2 * n * (n + 1) // 5, _log(rng, 20, 240)),
                "tau": rng.choice([1e-5, 1e-6])}
    precision = "fp64" if kind in ("semicanonical", "df") else rng.choice(["bf16x3", "bf16x3", "tf32x3", "fp64"])
    if kind == "host" and precision == "fp64":
        precision = "bf16x3"
    # no drawn case is dearer than the largest listed one of its kind
    most = _pair_work(24, 372, 1200)
    most = {"gradient": most if precision != "fp64" else most // 8}.get(
        kind, most if precision == "fp64" else _pair_work(24, 1214, 3400))
    while True:
        nC, nA, nV = _log(rng, 4, 40), rng.randint(0, 6), _log(rng, 40, 1214)
        naux = int(rng.uniform(2.6, 3.4) * (nC + nA + nV))
        if kind in ("semicanonical", "df"):
            if nV <= 372 and naux <= 1200:
                break
        elif _pair_work(nC, nV, naux) <= most // (2 if precision == "tf32x3" else 1):
            break
    ext = kind in ("energy", "gradient") and nA > 0 and rng.random() < 0.25
    c = _case("", kind, nC, nA, nV, naux, precision, rng.choice([0.1, 0.5, 0.5, 1.0]), ext)
    del c["name"]
    return c


# ------------------------------------ inputs ------------------------------------

def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + k) % (1 << 62))


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=F8).cuda()


def _decay(naux, scale):
    return (scale * torch.exp(-0.02 * torch.arange(naux, dtype=F8, device="cuda")))[:, None, None]


def _energies(rng, nC, nA, nV):
    return [rng.uniform(-2.0, -0.3, nC), rng.uniform(-0.2, 0.1, nA), rng.uniform(0.05, 5.0, nV)]


def _state(rng, nA):
    """Density and opposite-spin cumulant of the active space."""
    if nA == 0:
        return None, None
    d = rng.uniform(-1.0, 1.0, nA)
    d -= d.mean()
    d /= max(1.0, np.abs(d).max())
    U = np.linalg.qr(rng.standard_normal((nA, nA)))[0]
    L = rng.uniform(-0.05, 0.05, (nA,) * 4)
    L = L + L.transpose(2, 1, 0, 3)
    L = L + L.transpose(0, 3, 2, 1)
    L = (L + L.transpose(1, 0, 3, 2)) / 8.0
    G = (U * (1.0 + d)) @ U.T
    return _cuda(0.5 * (G + G.T)), _cuda(L)


def _cumulant3(nA, g):
    """Spin-orbital three-body cumulant: spin conserving, antisymmetric in each triple, Hermitian."""
    n2 = 2 * nA
    R = 0.04 * (torch.rand((n2,) * 6, dtype=F8, device="cuda", generator=g) - 0.5)
    al = (torch.arange(n2, device="cuda") % 2 == 0).long()
    na = al[:, None, None] + al[None, :, None] + al[None, None, :]
    R = R * (na[:, :, :, None, None, None] == na)
    for o in (0, 3):
        a, b, c = o, o + 1, o + 2
        R = (R - R.transpose(a, b)) / 2.0
        R = (R + R.movedim((a, b, c), (b, c, a)) + R.movedim((a, b, c), (c, a, b))) / 3.0
    return 0.5 * (R + R.permute(3, 4, 5, 0, 1, 2)).contiguous()


def _molecule(nC, nA, nV, naux, seed, ext=False):
    """Inputs of the energy on the GPU: (B, eps, gamma1, lambda2, lambda3, f1)."""
    rng = np.random.default_rng([int(seed), nC, nA, nV, naux])
    B = torch.randn((naux, nC + nA, nA + nV), dtype=F8, device="cuda", generator=_gen(seed, naux + 7 * nV + nC))
    if nA:
        aa = B[:, nC:, :nA]
        B[:, nC:, :nA] = torch.triu(aa) + torch.triu(aa, 1).transpose(1, 2)
    B *= _decay(naux, 0.3)
    eps = _cuda(np.concatenate([np.sort(e) for e in _energies(rng, nC, nA, nV)]))
    G, L = _state(rng, nA)
    l3 = f1 = None
    if ext:
        l3 = _cumulant3(nA, _gen(seed, 3))
        f1 = _cuda(rng.uniform(-0.05, 0.05, (nC + nA, nA + nV)))
        f1[nC:, :nA] = 0.0
    return B, eps, G, L, l3, f1


def _sizes(case):
    return case["ncore"], case["nactive"], case["nvirt"], case["naux"]


def _batch_sizes(case):
    r = random.Random(case["sizes_seed"])
    out = []
    for _ in range(case["molecules"]):
        nC, nA, nV = r.randint(8, 40), r.randint(2, 6), r.randint(100, 600)
        out.append((nC, nA, nV, int(round(3.2 * (nC + nA + nV)))))
    return out


def _batch_inputs(case, seed):
    return [_molecule(*sz, seed=int(seed) * 64 + k) for k, sz in enumerate(_batch_sizes(case))]


def _fock_inputs(case, seed):
    nC, nA, nV, naux = _sizes(case)
    n = nC + nA + nV
    rng = np.random.default_rng([int(seed), n, naux])
    B = torch.randn((naux, n, n), dtype=F8, device="cuda", generator=_gen(seed, n))
    B = 0.5 * (B + B.transpose(1, 2))
    B *= _decay(naux, 0.05)
    R = rng.uniform(-0.05, 0.05, (n, n))
    h = np.diag(np.concatenate(_energies(rng, nC, nA, nV))) + 0.5 * (R + R.T)
    return (_cuda(h), B) + _state(rng, nA)


def _df_inputs(case, seed):
    nC, nA, nV, naux = _sizes(case)
    n = nC + nA + nV
    a = torch.randn((naux, n, n), dtype=F8, device="cuda", generator=_gen(seed, n + 1))
    a = 0.5 * (a + a.transpose(1, 2))
    a *= _decay(naux, 0.3)
    C = torch.linalg.qr(torch.randn((n, n), dtype=F8, device="cuda", generator=_gen(seed, n + 2)))[0].contiguous()
    W = torch.randn((naux, naux), dtype=F8, device="cuda", generator=_gen(seed, n + 3))
    J = W @ W.T / naux + 0.1 * torch.eye(naux, dtype=F8, device="cuda")
    return a, C, (0.5 * (J + J.T)).contiguous()


def _eri_factors(case, seed):
    n, k = case["nbf"], case["nfac"]
    F = torch.randn((k, n, n), dtype=F8, device="cuda", generator=_gen(seed, 11 * n + k))
    F = 0.5 * (F + F.transpose(1, 2))
    F *= _decay(k, 0.3)
    return F


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        mols = _batch_inputs(case, seed)
        plan = pk.Batch(_batch_sizes(case), precision=case["precision"])
        return case, plan, [m[:4] for m in mols], [case["s"]] * len(mols)
    if kind == "cholesky":
        return case, None, _eri_factors(case, seed), None
    if kind == "df":
        return case, None, _df_inputs(case, seed), None
    if kind == "semicanonical":
        return case, pk.SemicanonicalPlan(*_sizes(case)), _fock_inputs(case, seed), None
    mol = _molecule(*_sizes(case), seed=seed, ext=case["ext"])
    plan = pk.Plan(*_sizes(case), precision=case["precision"], grad=kind == "gradient",
                   host_io=kind == "host")
    if kind == "host":
        host = []
        for t in mol[:4]:
            host.append(None if t is None else torch.empty(t.shape, dtype=F8, pin_memory=True).copy_(t))
        return case, plan, host, None
    return case, plan, mol, None


def run(state):
    case, plan, x, s = state
    kind = case["kind"]
    if kind == "energy":
        B, eps, G, L, l3, f1 = x
        return plan.energy(B, eps, G, L, case["s"], lambda3=l3, f1=f1)
    if kind == "gradient":
        B, eps, G, L, l3, f1 = x
        E, dB, deps, ds = plan.energy_grad(B, eps, G, L, case["s"], lambda3=l3, f1=f1)
        return {"energy": E, "dB": dB, "deps": deps, "ds": ds}
    if kind == "host":
        return plan.energy_host(*x, case["s"])
    if kind == "batch":
        return plan.energy(x, s)
    if kind == "semicanonical":
        out = plan.semicanonicalize(*x)
        return {k: v for k, v in out.items() if v is not None}
    if kind == "df":
        nC, nA, nV, _ = _sizes(case)
        return pk.df_mo_transform(*x, p0=0, np_=nC + nA, q0=nC, nq=nA + nV)
    return pk.cd_factors(x, tau=case["tau"])


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [_energy_work(*sz) for sz in _batch_sizes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if kind == "cholesky":
        n, k = case["nbf"], case["nfac"]
        N = n * (n + 1) // 2  # distinct pairs; the rank is at most nfac
        return {"bytes": 16 * k * n * n, "flops": 4 * min(k, N) ** 2 * N}
    nC, nA, nV, naux = _sizes(case)
    nH, nP, n = nC + nA, nA + nV, nC + nA + nV
    if kind == "semicanonical":
        rot = 2 * naux * nH * nP * (min(nH, nP) + nP)
        return {"bytes": 8 * (naux * n * n + naux * nH * nP + 3 * n * n),
                "flops": naux * n * n * (2 + nH) + 9 * nV ** 3 + rot}
    if kind == "df":
        # holes first (nH < nbf), then the metric's root and its product
        return {"bytes": 8 * (naux * n * n + naux * nH * nP + naux * naux),
                "flops": 2 * naux * nH * n * (n + nP) + naux ** 3 // 3 + naux * naux * nH * nP}
    w = _energy_work(nC, nA, nV, naux)
    if kind == "gradient":  # each product's two adjoints, and dB written
        return {"bytes": 2 * w["bytes"], "flops": 3 * w["flops"]}
    return w


def _energy_work(nC, nA, nV, naux):
    """B read once; the pair products of F1 (i <= j) and F2."""
    return {"bytes": 8 * (naux * (nC + nA) * (nA + nV) + 5),
            "flops": _pair_work(nC, nV, naux) + 2 * nC * nA * naux * nV * nV}


# ------------------------- the same outputs in plain FP64 torch -------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        if work(case)["flops"] > 8e12:
            return None
        with torch.no_grad():
            return torch.stack([_energy(m, sz, case["s"]) for m, sz in
                                zip(_batch_inputs(case, seed), _batch_sizes(case))])
    if kind == "cholesky":
        return _exact_cholesky(_eri_factors(case, seed), case["tau"])
    if kind == "df":
        nC, nA, nV, naux = _sizes(case)
        a, C, J = _df_inputs(case, seed)
        Z = (C[:, :nC + nA].T @ a @ C[:, nC:]).reshape(naux, -1)
        return torch.linalg.solve_triangular(torch.linalg.cholesky(J), Z, upper=False).reshape(
            naux, nC + nA, nA + nV)
    if kind == "semicanonical":
        return _exact_semicanonical(case, *_fock_inputs(case, seed))
    mol = _molecule(*_sizes(case), seed=seed, ext=case["ext"])
    if kind in ("energy", "host"):
        with torch.no_grad():
            return _energy(mol, _sizes(case), case["s"])
    B, eps = mol[0].requires_grad_(True), mol[1].requires_grad_(True)
    s = torch.tensor(case["s"], dtype=F8, device="cuda", requires_grad=True)
    E = _energy((B, eps) + mol[2:], _sizes(case), s)
    dB, deps, ds = torch.autograd.grad(E[4], (B, eps, s))
    return {"energy": E.detach(), "dB": dB, "deps": deps, "ds": ds.reshape(1)}


def _rt(D, s):
    """(1 - e^{-s D^2}) / D with its limit s D at 0."""
    z = D == 0
    return torch.where(z, s * D, -torch.expm1(-s * D * D) / torch.where(z, torch.ones_like(D), D))


def _rv(D, s):
    return 1.0 + torch.exp(-s * D * D)


def _energy(mol, sizes, s):
    """[E_CCVV, E_CAVV, E_CCAV, E_active, E_total] (arXiv:1603.00561, Tables 1 and 2)."""
    B, eps, G, L, l3, f1 = mol
    nC, nA, nV, _ = sizes
    eC, eA, eV = eps[:nC], eps[nC:nC + nA], eps[nC + nA:]
    rows = B[:, :, nA:].permute(1, 2, 0).contiguous()     # [hole, virtual, Q]
    vv = eV[:, None] + eV[None, :]
    zero = torch.zeros((), dtype=F8, device=B.device)
    f1_ = zero
    for i in range(nC):
        for j in range(i, nC):
            v = rows[i] @ rows[j].T
            e = torch.sum(v * (2.0 * v - v.T) * _rt(eC[i] + eC[j] - vv, 2.0 * s))
            f1_ = f1_ + (e if i == j else 2.0 * e)
    f2 = f3 = act = zero
    if nA:
        for m in range(nC):                                # X_u[e,f] = (me|uf)
            X = rows[m] @ rows[nC:].transpose(1, 2)
            D = eC[m] + eA[:, None, None] - vv
            A = torch.einsum("uv,uef->vef", G, X * _rv(D, s))
            f2 = f2 + torch.sum(A * (2.0 * X - X.transpose(1, 2)) * _rt(D, s))
        Z = torch.einsum("Qme,Qnu->umne", B[:, :nC, nA:], B[:, :nC, :nA])
        D = eC[:, None, None] + eC[None, :, None] - eV - eA[:, None, None, None]
        H = 2.0 * torch.eye(nA, dtype=F8, device=B.device) - G
        f3 = torch.sum(torch.einsum("uv,vmne->umne", H, Z * _rv(D, s))
                       * (2.0 * Z - Z.transpose(1, 2)) * _rt(D, s))
        act = _active(B, eps, G, L, l3, f1, s, nC, nA)
    elif f1 is not None:
        D = eC[:, None] - eV[None, :]
        act = 2.0 * torch.sum(f1 * f1 * _rv(D, s) * _rt(D, s))
    return torch.stack([f1_, f2, f3, act, f1_ + f2 + f3 + act])


def _active(B, eps, G, L, l3, f1, s, nC, nA):
    """Terms A-E and G-K of Table 1 and F4-F8 of Table 2 in spin orbitals 2 p + sigma."""
    dev = B.device
    nH, nP = B.shape[1], B.shape[2]
    two = lambda k: torch.arange(2 * k, device=dev)
    eH, eP = eps[:nH].repeat_interleave(2), eps[nC:].repeat_interleave(2)
    allH, allP = two(nH), two(nP)
    aH, aP = allH[2 * nC:], allP[:2 * nA]
    c, ah, ap, vv = slice(0, 2 * nC), slice(2 * nC, None), slice(0, 2 * nA), slice(2 * nA, None)

    def block(I, J, P, R):
        """V = <IJ||PR>, its amplitudes T and its modified integrals W."""
        hi, hj = I[::2] // 2, J[::2] // 2
        pa, pb = P[::2] // 2, R[::2] // 2
        at = lambda h, p: B[:, h[0]:h[-1] + 1, p[0]:p[-1] + 1]
        i, j, a, b = (torch.arange(len(x), device=dev) for x in (I, J, P, R))
        si, sj = (i % 2)[:, None, None, None], (j % 2)[:, None, None]
        sa, sb = (a % 2)[:, None], b % 2
        up = lambda t: t.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)
        V = (up(torch.einsum("Qia,Qjb->ijab", at(hi, pa), at(hj, pb))) * ((si == sa) & (sj == sb))
             - up(torch.einsum("Qib,Qja->ijab", at(hi, pb), at(hj, pa))) * ((si == sb) & (sj == sa)))
        D = eH[I][:, None, None, None] + eH[J][:, None, None] - eP[P][:, None] - eP[R]
        inner = ((I >= 2 * nC)[:, None, None, None] & (J >= 2 * nC)[:, None, None]
                 & (P < 2 * nA)[:, None] & (R < 2 * nA))
        return torch.where(inner, torch.zeros_like(V), V * _rt(D, s)), V * _rv(D, s)

    T1, W1 = block(allH, aH, allP, aP)     # (H, A | P, A)
    T2, W2 = block(allH, allH, aP, aP)     # (H, H | A, A)
    T3, W3 = block(aH, aH, allP, allP)     # (A, A | P, P)
    g = torch.kron(G / 2.0, torch.eye(2, dtype=F8, device=dev))
    h = torch.eye(2 * nA, dtype=F8, device=dev) - g

    def gam(X, ax):                        # gamma over a hole axis
        X = X.movedim(ax, 0)
        return torch.cat([X[c], torch.tensordot(g, X[ah], dims=([1], [0]))]).movedim(0, ax)

    def eta(X, ax):                        # eta over a particle axis
        X = X.movedim(ax, 0)
        return torch.cat([torch.tensordot(h, X[ap], dims=([1], [0])), X[vv]]).movedim(0, ax)

    n2 = 2 * nA
    lam = torch.zeros((n2,) * 4, dtype=F8, device=dev)
    A, Bt = slice(0, None, 2), slice(1, None, 2)
    same = L - L.permute(0, 1, 3, 2)
    lam[A, A, A, A] = same
    lam[Bt, Bt, Bt, Bt] = same
    lam[A, Bt, A, Bt] = L
    lam[Bt, A, Bt, A] = L.permute(1, 0, 3, 2)
    lam[A, Bt, Bt, A] = -L.permute(0, 1, 3, 2)
    lam[Bt, A, A, Bt] = -L.permute(1, 0, 2, 3)

    # singles: T1 and the modified Fock block (Eqs. (12), (14))
    eAs = eH[2 * nC:]
    S = torch.einsum("ux,iuax,ux->ia", eAs[None, :] - eAs[:, None], T1, g)
    D1 = eH[:, None] - eP
    inner = (allH >= 2 * nC)[:, None] & (allP < n2)
    F1 = torch.zeros_like(S)
    if f1 is not None:
        F1 = f1.repeat_interleave(2, 0).repeat_interleave(2, 1) * (allH[:, None] % 2 == allP % 2)
        F1 = torch.where(inner, torch.zeros_like(F1), F1)
    t = torch.where(inner, torch.zeros_like(S), (F1 + S) * _rt(D1, s))
    g1 = torch.exp(-s * D1 * D1)
    f = F1 * (1.0 + g1) + S * g1

    es = torch.einsum
    out = torch.sum(gam(f, 0) * eta(t, 1))                                                     # A
    out = out + 0.5 * torch.sum(es("xyev,ue->xyuv", W3[:, :, vv, ap], t[ah, vv]) * lam.permute(2, 3, 0, 1))   # B
    out = out - 0.5 * torch.sum(es("myuv,mx->xyuv", W1[c, :, ap, :], t[c, ap]) * lam.permute(2, 3, 0, 1))     # C
    out = out + 0.5 * torch.sum(es("xe,uvey->uvxy", f[ah, vv], T3[:, :, vv, ap]) * lam)                       # D
    out = out - 0.5 * torch.sum(es("mv,umxy->uvxy", f[c, ap], T2[ah, c]) * lam)                               # E
    out = out + 0.125 * torch.sum(es("xycd,uvcd->uvxy", W3, eta(eta(T3, 2), 3)) * lam)                        # G
    out = out + 0.125 * torch.sum(es("kluv,klxy->uvxy", W2, gam(gam(T2, 0), 1)) * lam)                        # H
    out = out + torch.sum(es("jxbu,jvby->uvxy", W1, eta(gam(T1, 0), 2)) * lam)                                # I
    out = out + 0.25 * es("xuyv,xy,uv->", es("xuef,yvef->xuyv", W3[:, :, vv, vv], T3[:, :, vv, vv]), g, g)    # F4
    out = out + 0.25 * es("vyux,uv,xy->", es("mnvy,mnux->vyux", W2[c, c], T2[c, c]), h, h)                    # F5
    out = out + es("xvyu,xy,uv->", es("mxev,myeu->xvyu", W1[c, :, vv, :], T1[c, :, vv, :]), g, h)             # F6
    out = out + 0.5 * es("yzvwxu,yw,zx,uv->", es("yzve,wxue->yzvwxu", W3[:, :, ap, vv], T3[:, :, ap, vv]), g, g, h)  # F7
    out = out + 0.5 * es("wvyzux,wz,uv,xy->", es("mwvy,mzux->wvyzux", W1[c, :, ap, :], T1[c, :, ap, :]), g, h, h)    # F8
    if l3 is not None:
        out = out + 0.25 * torch.sum(es("mzuv,mwxy->uvwxyz", W1[c, :, ap, :], T1[c, :, ap, :]) * l3)          # J
        out = out + 0.25 * torch.sum(es("xywe,uvez->uvwxyz", W3[:, :, ap, vv], T3[:, :, vv, ap]) * l3)        # K
    return out


def _exact_semicanonical(case, h, B, G, L):
    nC, nA, nV, naux = _sizes(case)
    nH, n = nC + nA, nC + nA + nV
    D = torch.zeros((nH, nH), dtype=F8, device="cuda")
    D[range(nC), range(nC)] = 2.0
    if nA:
        D[nC:, nC:] = G
    X = B[:, :, :nH] @ D
    w = (X[:, :nH].diagonal(dim1=1, dim2=2)).sum(1)
    K = X.permute(1, 0, 2).reshape(n, -1) @ B[:, :nH].reshape(-1, n)
    f = h + torch.tensordot(w, B, dims=1) - 0.5 * K
    f = 0.5 * (f + f.T)
    U = torch.zeros_like(f)
    for lo, hi in ((0, nC), (nC, nH), (nH, n)):
        if hi > lo:
            V = torch.linalg.eigh(f[lo:hi, lo:hi])[1]
            k = V.abs().argmax(0)
            U[lo:hi, lo:hi] = V * torch.sign(V[k, torch.arange(hi - lo, device="cuda")])
    fs = U.T @ f @ U
    f1 = fs[:nH, nC:].clone()
    f1[nC:, :nA] = 0.0
    out = {"eps": fs.diagonal().clone(), "B": U[:nH, :nH].T @ B[:, :nH, nC:] @ U[nC:, nC:], "f1": f1, "U": U}
    if nA:
        A = U[nC:nH, nC:nH]
        out["gamma1"] = A.T @ G @ A
        out["lambda2"] = torch.einsum("au,bv,cx,dy,abcd->uvxy", A, A, A, A, L)
    return out


def _exact_cholesky(F, tau):
    """Outer-product Cholesky with diagonal pivoting; of equal pairs (p, q), (q, p) the upper one."""
    k, n, _ = F.shape
    M = F.reshape(k, n * n)
    d = (M * M).sum(0)
    upper = torch.triu(torch.ones((n, n), dtype=torch.bool, device="cuda")).reshape(-1)
    L = torch.zeros((min(k, n * n), n * n), dtype=F8, device="cuda")
    r = 0
    while r < len(L):
        p = int(torch.where(upper, d, torch.full_like(d, -1.0)).argmax())
        if float(d[p]) < tau:
            break
        L[r] = (M[:, p] @ M - L[:r, p] @ L[:r]) / torch.sqrt(d[p])
        d = d - L[r] * L[r]
        d[p] = 0.0
        r += 1
    return L[:r].reshape(r, n, n)
