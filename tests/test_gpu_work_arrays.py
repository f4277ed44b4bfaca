"""The input builders in little memory: work arrays and plans without room for the digits of
the products on the tensor cores. Fewer bytes change the route of the products, not what they
are: the results agree within the FP64 bar of their other tests.
"""
import ctypes as C

import numpy as np
import pytest

from dsrg_synth import make_ao_problem, make_eri_factors, make_fock_problem

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
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64).cuda()


def _leave_free(torch, nbytes):
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - nbytes, dtype=torch.uint8, device="cuda")


def _df(lib, torch, p, np_, q0, nq, work_bytes):
    """(status, B) of a call with a work array of work_bytes inside guarded memory."""
    ao3, Cm, J = _dev(p.ao3), _dev(p.C), _dev(p.metric)
    out = torch.full((p.naux, np_, nq), 777.0, dtype=torch.float64, device="cuda")
    work = torch.full((work_bytes + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    ptr = lambda t: C.c_void_p(t.data_ptr())
    st = lib.dsrg_df_mo_transform(ptr(ao3), ptr(Cm), ptr(J), p.nbf, p.C.shape[1], p.naux, 0, np_, q0, nq, ptr(out),
                                  ptr(work), work_bytes, C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert (work[work_bytes:] == 0x5A).all()
    return st, out.cpu().numpy()


@pytest.mark.parametrize("nbf,naux,np_,nq", [(150, 500, 33, 117), (130, 700, 5, 125)])
def test_df_transform_in_any_work_array(pk, nbf, naux, np_, nq):
    """From the least size on, the former size (64 bytes past the matrices) among them: sizes that
    leave no room, room for a few problems or a few row blocks of a product, and all of it."""
    import torch
    from paper_1603_00561_gb300 import _native
    lib = _native.load()
    p = make_ao_problem(nbf, nbf, naux, seed=12)
    least = lib.dsrg_df_mo_transform_min_work_bytes(nbf, naux, np_, nq)
    most = lib.dsrg_df_mo_transform_work_bytes(nbf, naux, np_, nq)
    assert least == 8 * (naux * np_ * nbf + naux * np_ * nq + 2 * naux * naux) + 64 < most
    st, ref = _df(lib, torch, p, np_, nbf - nq, nq, most)
    assert st == _native.OK
    for f in (0.0, 1e-4, 0.003, 0.02, 0.05, 0.1, 0.2, 0.4, 0.7, 0.95, 1.1):
        st, B = _df(lib, torch, p, np_, nbf - nq, nq, least + int(f * (most - least)) // 8 * 8)
        assert st == _native.OK
        assert np.abs(B - ref).max() <= 1e-12 * np.abs(ref).max(), f
    st, _ = _df(lib, torch, p, np_, nbf - nq, nq, least - 8)
    assert st == _native.ERR_INVALID_ARG


def test_df_transform_with_little_free_memory(pk):
    """The Python call allocates the work array itself."""
    import torch
    p = make_ao_problem(400, 400, 500, seed=13)
    ao3, Cm, J = _dev(p.ao3), _dev(p.C), _dev(p.metric)
    ref = pk.df_mo_transform(ao3, Cm, J, 0, 20, 20, 380).clone()
    from paper_1603_00561_gb300 import _native
    lib = _native.load()
    least = lib.dsrg_df_mo_transform_min_work_bytes(400, 500, 20, 380)
    most = lib.dsrg_df_mo_transform_work_bytes(400, 500, 20, 380)
    out = ref.numel() * 8
    assert most > least + (300 << 20)
    filler = _leave_free(torch, least + out + (200 << 20))
    try:
        B = pk.df_mo_transform(ao3, Cm, J, 0, 20, 20, 380)
    finally:
        del filler
        torch.cuda.empty_cache()
    assert (B - ref).abs().max() <= 1e-12 * ref.abs().max()


@pytest.mark.parametrize("n,nfac", [(3, 4), (30, 120)])
def test_cholesky_in_a_work_array_of_the_former_size(pk, n, nfac):
    """8 n^2 + 88 bytes: the same vectors, bit for bit, as with all that the call asks for."""
    import torch
    from paper_1603_00561_gb300 import _native
    lib = _native.load()
    F = _dev(make_eri_factors(n, nfac, seed=2))
    ref = pk.cd_factors(F, 1e-7)
    ptr = lambda t: C.c_void_p(t.data_ptr())
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    for wb, want in ((8 * n * n + 88, _native.OK), (8 * n * n + 80, _native.ERR_INVALID_ARG)):
        L = torch.zeros((n * n, n, n), dtype=torch.float64, device="cuda")
        work = torch.full((wb + 512,), 0x5A, dtype=torch.uint8, device="cuda")
        rank = C.c_int32(-1)
        assert lib.dsrg_cd_factors(ptr(F), nfac, n, 1e-7, n * n, ptr(L), C.byref(rank), ptr(work), wb, stream) == want
        assert (work[wb:] == 0x5A).all()
        if want == _native.OK:
            assert rank.value == ref.shape[0] and torch.equal(L[: rank.value], ref)


def test_semicanonical_plan_with_little_free_memory(pk):
    """Without room for digits and partial exchange matrices the plan is made all the same."""
    import torch
    nC, nA, nV, Q = 8, 2, 200, 1500
    n, nH, nP = nC + nA + nV, nC + nA, nA + nV
    p = make_fock_problem(nC, nA, nV, Q, seed=5)
    args = [_dev(x) for x in (p.h, p.Bfull, p.gamma1, p.lambda2)]
    sc = pk.SemicanonicalPlan(nC, nA, nV, Q)
    ref = sc.semicanonicalize(*args)
    f = sc.fock(*args[:3])
    sc.close()
    # the arrays that the plan is documented to need, in 2 MiB granules, and its outputs
    need = 8 * (Q * n * (nH + 1) + 2 * Q * nH * nP + 7 * n * n) + (40 << 20)
    out = 8 * (Q * nH * nP + 3 * n * n) + (60 << 20)
    filler = _leave_free(torch, need + out)
    try:
        sc = pk.SemicanonicalPlan(nC, nA, nV, Q)
        got = sc.semicanonicalize(*args)
        f2 = sc.fock(*args[:3])
        sc.sync()
        sc.close()
    finally:
        del filler
        torch.cuda.empty_cache()
    assert (f2 - f).abs().max() <= 1e-12 * f.abs().max()
    assert (got["eps"] - ref["eps"]).abs().max() <= 1e-12 * f.abs().max()
    assert (got["B"] - ref["B"]).abs().max() <= 1e-9 * ref["B"].abs().max()
