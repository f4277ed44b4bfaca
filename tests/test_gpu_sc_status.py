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
