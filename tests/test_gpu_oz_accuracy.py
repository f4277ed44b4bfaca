"""Products of graded operands: the digit products (csrc/oz_gemm.cu) may not lose what a
chain of FP64 FMAs keeps.

A chain of K FMAs is within K 2^-53 sum_k |a_k b_k| of the exact sum (first order),
whatever the sizes of its terms. Every bar below is that bound, taken element by
element from the inputs and carried through what follows by first order, plus
the roundings of the steps around it; factors of 2 cover the second order and the
rounding of the reference. Inputs: two weakly coupled fragments, auxiliary
functions that decay in opposite directions, badly scaled auxiliary functions.
"""
import numpy as np
import pytest

from dsrg_synth import make_ao_problem, make_problem

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def pk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1603_00561_gb300 as pk
    pk.build()
    return pk


def _dev(x):
    import torch
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64).cuda()


def _pair_reference(B, eps, s, nC, nA):
    """Pair energies e_ij = sum_ab v_ab (2 v_ab - v_ba) R_ab in long double, and the bound of
    an FP64 evaluation whose integrals are FMA chains."""
    Q, _, nP = B.shape
    L = B[:, :nC, nA:].astype(np.longdouble)
    e, bar = np.zeros((nC, nC)), np.zeros((nC, nC))
    ec, ev = eps[:nC].astype(np.longdouble), eps[nC + nA:].astype(np.longdouble)
    for i in range(nC):
        for j in range(nC):
            v = L[:, i].T @ L[:, j]
            S = (np.abs(L[:, i]).T @ np.abs(L[:, j])).astype(float)
            D = ec[i] + ec[j] - ev[:, None] - ev[None, :]
            R = -np.expm1(-2 * np.longdouble(s) * D * D) / D
            e[i, j] = float(np.sum(v * (2 * v - v.T) * R))
            av, aR, d = np.abs(v).astype(float), np.abs(R).astype(float), (Q + 1) * U * S
            # the integrals, and 64 roundings of the regulator, the products and their sum
            bar[i, j] = np.sum(aR * (4 * av * d + av * d.T + av.T * d))
            bar[i, j] += 64 * U * np.sum(aR * av * (2 * av + av.T))
    return e, 2 * bar


def _inputs(kind, nC, nA, nV, Q, seed):
    p = make_problem(nC, nA, nV, Q, s=0.5, seed=seed, b_decay=0.0)
    B = p.B.copy()
    q = np.arange(Q)
    if kind == "fragments":
        # core orbital i and every orbital pair with it on fragment i % 2: its own half of the
        # auxiliary functions, 1e-10 on the other's
        for i in range(nC):
            B[(q < Q // 2) == (i % 2 == 1), i] *= 1e-10
    elif kind == "opposite":
        for i in range(nC):
            B[:, i] *= np.exp(-0.05 * (q if i % 2 else q[::-1]))[:, None]
    elif kind == "one column":
        # virtual a large only on auxiliary function a, everything else 1e-9 of it
        B[:, :, nA:] *= np.where((q[:, None] % nV) == np.arange(nV)[None], 1.0, 1e-9)[:, None, :]
    return p, B


@pytest.mark.parametrize("kind", ["fragments", "opposite", "one column"])
@pytest.mark.parametrize("nC,nA,nV,Q", [(3, 0, 70, 2), (4, 0, 33, 31), (4, 2, 129, 300)])
def test_pair_energies_of_graded_factors(pk, kind, nC, nA, nV, Q):
    p, B = _inputs(kind, nC, nA, nV, Q, 7)
    plan = pk.Plan(nC, nA, nV, Q, precision="fp64")
    e = plan.pair_energies(_dev(B), _dev(p.eps), p.s).cpu().numpy()
    plan.sync()
    ref, bar = _pair_reference(B, p.eps, p.s, nC, nA)
    assert (np.abs(e - ref) <= bar).all(), (np.abs(e - ref) / bar).max()


def test_fock_matrix_of_graded_factors(pk):
    """The exchange product over (Q, r): orbital p decays along Q, orbital q the other way."""
    nC, nA, nV, Q = 12, 2, 100, 420
    n = nC + nA + nV
    r = np.random.default_rng(3)
    B = r.standard_normal((Q, n, n))
    dec = np.exp(-0.08 * np.arange(Q))
    half = np.arange(n) % 2 == 1
    w = np.where(half[None, :], dec[:, None], dec[::-1, None])
    B *= np.maximum(w[:, :, None], 1e-13) * np.maximum(w[:, None, :], 1e-13)
    B = 0.5 * (B + B.transpose(0, 2, 1))
    G = np.diag([1.25, 0.75])
    h = np.zeros((n, n))
    sc = pk.SemicanonicalPlan(nC, nA, nV, Q)
    f = sc.fock(_dev(h), _dev(B), _dev(G)).cpu().numpy()
    D = np.zeros(n)
    D[:nC], D[nC:nC + nA] = 2.0, np.diag(G)
    L, DL = B.astype(np.longdouble), D.astype(np.longdouble)
    wq = np.einsum("Qrr,r->Q", L, DL)
    J = np.einsum("Qpq,Q->pq", L, wq)
    nH = nC + nA
    X = (L[:, :, :nH] * DL[None, None, :nH]).transpose(1, 0, 2).reshape(n, -1)
    Y = L[:, :nH, :].transpose(2, 0, 1).reshape(n, -1)
    ref = (J - 0.5 * X @ Y.T).astype(float)
    aw = np.einsum("Qrr,r->Q", np.abs(B), D)
    bar = ((Q + n + 4) * U * np.einsum("Qpq,Q->pq", np.abs(B), aw)
           + (Q * nH + 4) * U * 0.5 * np.abs(X).astype(float) @ np.abs(Y).astype(float).T)
    bar = bar + bar.T  # f is symmetrised
    assert (np.abs(f - ref) <= 2 * bar).all(), (np.abs(f - ref) / (2 * bar)).max()


@pytest.mark.parametrize("nbf,nmo,naux,np_,nq", [(150, 149, 500, 75, 147), (131, 131, 257, 64, 129)])
def test_df_factors_do_not_depend_on_the_scale_of_the_auxiliaries(pk, nbf, nmo, naux, np_, nq):
    """With T a diagonal of powers of two, (T ao3, T J T) has the same factors as (ao3, J): L
    becomes T L, L^-1 becomes L^-1 T^-1, all exactly."""
    p = make_ao_problem(nbf, nmo, naux, seed=11)
    T = 2.0 ** np.random.default_rng(5).integers(-20, 21, naux)
    args = (0, np_, nmo - nq, nq)
    B = pk.df_mo_transform(_dev(p.ao3), _dev(p.C), _dev(p.metric), *args).cpu().numpy()
    Bt = pk.df_mo_transform(_dev(p.ao3 * T[:, None, None]), _dev(p.C),
                            _dev(p.metric * T[:, None] * T[None, :]), *args).cpu().numpy()
    # both sides within the chains' bounds of the three products (and of L^-1, the same
    # up to the scales) of one and the same number
    C0, C1 = np.abs(p.C[:, :np_]), np.abs(p.C[:, nmo - nq:])
    Li = np.abs(np.linalg.inv(np.linalg.cholesky(p.metric)))
    LL = Li @ np.abs(np.linalg.cholesky(p.metric)) @ Li
    Z = np.einsum("mp,Pmn,nq->Ppq", C0, np.abs(p.ao3), C1, optimize=True).reshape(naux, -1)
    bar = U * ((2 * nbf + naux) * Li + 2 * naux * LL) @ Z
    assert (np.abs(Bt - B).reshape(naux, -1) <= 2 * 2 * bar).all()
    mo = np.einsum("mp,Pmn,nq->Ppq", p.C[:, :np_], p.ao3, p.C[:, nmo - nq:], optimize=True)
    ref = np.linalg.solve(np.linalg.cholesky(p.metric), mo.reshape(naux, -1))
    assert np.abs(B.reshape(naux, -1) - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("decay", [0.0, 0.1])
def test_df_of_a_diagonal_metric(pk, decay):
    """L^-1 diagonal: B[Q] = 2^-k_Q Z[Q] with Z = C^T ao3 C, element by element; with the AO
    functions graded one way in ao3 and the other way in C."""
    nbf, nmo, naux = 150, 140, 203
    r = np.random.default_rng(8)
    g = np.exp(-decay * np.arange(nbf))
    ao = r.standard_normal((naux, nbf, nbf))
    ao = 0.5 * (ao + ao.transpose(0, 2, 1)) * g[None, :, None] * g[None, None, :]
    C = r.standard_normal((nbf, nmo)) * g[::-1, None] * np.where(np.arange(nmo) % 2, 1.0, 1e-12)[None]
    k = r.integers(-30, 31, naux)
    B = pk.df_mo_transform(_dev(ao), _dev(C), _dev(np.diag(4.0 ** k))).cpu().numpy()
    aL, CL = ao.astype(np.longdouble), C.astype(np.longdouble)
    bound = 2 * (2 * nbf + naux + 4) * U
    for Q in range(0, naux, 29):
        ref = (CL.T @ aL[Q] @ CL).astype(float) * 2.0 ** -k[Q]
        bar = bound * (np.abs(C).T @ np.abs(ao[Q]) @ np.abs(C)) * 2.0 ** -k[Q]
        assert (np.abs(B[Q] - ref) <= bar).all(), (Q, (np.abs(B[Q] - ref) / bar).max())


@pytest.mark.parametrize("x,zero", [(0.75 * 2.0 ** -240, False), (0.75 * 2.0 ** -600, True),
                                    (3.0 * 2.0 ** -1072, True)])
@pytest.mark.parametrize("Q", [33, 129])
def test_scales_far_from_one(pk, x, zero, Q):
    """Integrals near the end of the FP64 range, and factors whose products underflow (2^-1072:
    below the normal range themselves)."""
    p = make_problem(2, 0, 65, Q, s=0.5, seed=1)
    B = np.full((Q, 2, 65), x)
    plan = pk.Plan(2, 0, 65, Q, precision="fp64")
    e = plan.pair_energies(_dev(B), _dev(p.eps), 0.5).cpu().numpy()
    plan.sync()
    if zero:
        assert (e == 0.0).all()
        return
    v = np.longdouble(x) ** 2 * Q
    eC, eV = p.eps[:2].astype(np.longdouble), p.eps[2:].astype(np.longdouble)
    for i in range(2):
        for j in range(2):
            D = eC[i] + eC[j] - eV[:, None] - eV[None, :]
            ref = np.sum(v * v * -np.expm1(-np.longdouble(1.0) * D * D) / D)
            assert abs(ref) > 1e-300
            assert abs(e[i, j] / ref - 1) <= 16 * 2.0 ** -52


def test_small_factor_times_large(pk):
    """Factors below the normal range against large ones: 2^-1060 2^1000, as in FP64."""
    nV, Q = 5, 3
    p = make_problem(2, 0, nV, Q, s=0.5, seed=2)
    B = np.zeros((Q, 2, nV))
    B[:, 0], B[:, 1] = 3.0 * 2.0 ** -1060, 5.0 * 2.0 ** 1000
    plan = pk.Plan(2, 0, nV, Q, precision="fp64")
    e = plan.pair_energies(_dev(B), _dev(p.eps), 0.5).cpu().numpy()
    plan.sync()
    v = np.longdouble(15.0 * Q * 2.0 ** -60)
    D = p.eps[:2].sum() - p.eps[2:][:, None] - p.eps[2:][None, :].astype(np.longdouble)
    ref = np.sum(v * v * -np.expm1(-D * D) / D)
    assert abs(e[0, 1] / ref - 1) <= 16 * 2.0 ** -52


def test_digits_at_the_most_negative(pk):
    """Values whose trailing digits are -128 (x = -1 - 2^-8 ... in the row scale): with the
    largest sums of digit products. Bar as test_gpu_oz_gemm.py."""
    # fixed-point 2^55 x with low byte 128 in every digit: (v - d) / 256 steps give d = -128
    v = 0
    for _ in range(6):
        v = (v << 8) - 128
    v += 127 << 48
    x = float(v) * 2.0 ** -55
    assert int(x * 2.0 ** 55) == v
    Q, nV = 900, 65
    p = make_problem(2, 0, nV, Q, s=0.5, seed=1)
    for sgn in (1.0, -1.0):
        plan = pk.Plan(2, 0, nV, Q, precision="fp64")
        e = plan.pair_energies(_dev(np.full((Q, 2, nV), sgn * x)), _dev(p.eps), 0.5).cpu().numpy()
        plan.sync()
        w = np.longdouble(x) ** 2 * Q
        eC, eV = p.eps[:2].astype(np.longdouble), p.eps[2:].astype(np.longdouble)
        D = eC[0] + eC[1] - eV[:, None] - eV[None, :]
        ref = np.sum(w * w * -np.expm1(-np.longdouble(1.0) * D * D) / D)
        assert abs(e[0, 1] / ref - 1) <= 16 * 2.0 ** -52


def test_infinite_rows_of_a_long_product(pk):
    """A row with an infinity (or a NaN) goes through FP64 FMAs element by element; of the
    exchange product's 31 000-long sums that is no reason to run into the bound of the
    kernels' waits. Rows and columns of the other orbitals are not touched."""
    import time
    import torch
    nC, nA, nV, Q = 24, 2, 130, 1200
    n = nC + nA + nV
    r = np.random.default_rng(9)
    B = torch.as_tensor(r.standard_normal((Q, n, n)) * np.exp(-0.02 * np.arange(Q))[:, None, None]).cuda()
    B = 0.5 * (B + B.transpose(1, 2)).contiguous()
    h, G = _dev(np.zeros((n, n))), _dev(np.diag([1.25, 0.75]))
    sc = pk.SemicanonicalPlan(nC, nA, nV, Q)
    good = sc.fock(h, B, G).clone()
    hit = [40, 41, 100]
    B[7, 30, hit] = float("inf")  # orbital 30 is virtual: only f[30, :] and f[:, hit] ...
    B[7, hit, 30] = float("inf")
    B[9, 50, 60] = float("nan")
    B[9, 60, 50] = float("nan")
    torch.cuda.synchronize()
    f = sc.fock(h, B, G)
    # J reads every pair: the pairs' own elements; K only hole columns, which are finite
    fine = torch.ones((n, n), dtype=torch.bool, device="cuda")
    for a, b in [(30, k) for k in hit] + [(50, 60)]:
        fine[a, b] = fine[b, a] = False
    assert not torch.isfinite(f[~fine]).any()
    assert torch.equal(f[fine], good[fine])
    # an infinity in a hole column: the whole row and column of that orbital, in K
    B[7, 3, 77] = B[7, 77, 3] = float("inf")
    torch.cuda.synchronize()
    t0 = time.time()
    f = sc.fock(h, B, G)
    torch.cuda.synchronize()
    assert time.time() - t0 < 1.0
    fine[77, :] = fine[:, 77] = False
    fine[3, :] = fine[:, 3] = False
    assert not torch.isfinite(f[77]).any()
    assert torch.equal(f[fine], good[fine])
