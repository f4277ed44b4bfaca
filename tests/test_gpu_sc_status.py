"""What the Fock build and the semicanonicalisation do when something is wrong: a
device-side wait that ran out, a Fock matrix that is not finite."""
import numpy as np
import pytest

from dsrg_synth import make_fock_problem

pytestmark = pytest.mark.gpu


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
    return None if x is None else torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64).cuda()


def test_a_wait_that_ran_out_is_reported(pk):
    """A product whose wait runs out leaves its tiles unwritten: f must not look valid, the next
    call that can wait says so, once, and the plan works again."""
    nC, nA, nV, Q = 4, 2, 50, 40
    p = make_fock_problem(nC, nA, nV, Q, seed=1)
    args = _dev(p.h), _dev(p.Bfull), _dev(p.gamma1)
    sc = pk.SemicanonicalPlan(nC, nA, nV, Q)
    from paper_1603_00561_gb300 import _native
    lib = _native.load()
    good = sc.fock(*args).cpu().numpy()
    sc.sync()
    for report in (sc.sync, lambda: sc.semicanonicalize(*args, _dev(p.lambda2))):
        assert lib.dsrg_sc_selftest_wait_timeout(sc.h) == _native.OK
        assert np.isnan(sc.fock(*args).cpu().numpy()).all()
        with pytest.raises(pk.DSRGError) as ei:
            report()
        assert ei.value.status == _native.ERR_TIMEOUT
        sc.sync()
        assert np.array_equal(sc.fock(*args).cpu().numpy(), good)
    out = sc.semicanonicalize(*args, _dev(p.lambda2))
    assert np.isfinite(out["eps"].cpu().numpy()).all()
    sc.close()


@pytest.mark.parametrize("block,bad", [("virtual", "nan"), ("virtual", "inf"), ("core", "nan"), ("all", "nan")])
def test_a_fock_matrix_that_is_not_finite(pk, block, bad):
    """Every output is written: the block's orbital energies and columns of U are not finite, those
    of the other blocks are what they are without it."""
    import ctypes as C
    import torch
    from paper_1603_00561_gb300 import _native
    lib = _native.load()
    nC, nA, nV, Q = 5, 2, 70, 40
    n, nH, nP = nC + nA + nV, nC + nA, nA + nV
    p = make_fock_problem(nC, nA, nV, Q, seed=3)
    B, G, L = _dev(p.Bfull), _dev(p.gamma1), _dev(p.lambda2)
    sc = pk.SemicanonicalPlan(nC, nA, nV, Q)
    good = sc.semicanonicalize(_dev(p.h), B, G, L)
    h = p.h.copy()
    lo, hi = {"virtual": (nH, n), "core": (0, nC), "all": (0, n)}[block]
    h[lo + 1, lo + 2] = h[lo + 2, lo + 1] = float(bad)
    if block == "all":
        h[:] = np.nan
    h = _dev(h)
    full = lambda *s: torch.full(s, 777.0, dtype=torch.float64, device="cuda")
    eps, Bo, f1, U, Go, Lo = full(n), full(Q, nH, nP), full(nH, nP), full(n, n), full(nA, nA), full(*(nA,) * 4)
    ptr = lambda t: C.c_void_p(t.data_ptr())
    st = lib.dsrg_semicanonicalize(sc.h, ptr(h), ptr(B), ptr(G), ptr(L), None, ptr(eps), ptr(Bo), ptr(f1),
                                   ptr(Go), ptr(Lo), None, ptr(U))
    assert st == _native.OK
    for t in (eps, Bo, f1, U, Go, Lo):
        assert not (t == 777.0).any()
    assert not torch.isfinite(eps[lo:hi]).any()
    blocks = [(0, nC), (nC, nH), (nH, n)] if block == "all" else [(lo, hi)]
    for a, b in blocks:
        assert torch.isnan(U[a:b, a:b]).any(dim=0).all()  # no column left at zero
    for a, b in [(0, nC), (nC, nH), (nH, n)]:
        if block != "all" and (a, b) != (lo, hi):
            assert torch.equal(eps[a:b], good["eps"][a:b])
            assert torch.equal(U[a:b, a:b], good["U"][a:b, a:b])
    sc.close()
