"""The active block at the edges of its kernels' tiles: terms J and K as products
with the antisymmetrised cumulant (16 x 16 tiles of triples x orbitals), the VV
adjoint (256 / nA^2 positions per CTA), the spin-restricted adjoints, the FP64
products in 16-, 32- and 64-wide tiles, and the FP32-pair adjoints of F1 and F2.

Bars as in the other tests: FP64 plans 1e-10, gradients of split plans 1e-5 of
the largest entry of each array.
"""
import numpy as np
import pytest

from dsrg_synth import make_problem
from oracle import dsrg as odsrg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1603_00561_gb300 as pk
    pk.build()
    return pk


CASES = [
    # nC, nA, nV, naux, s, seed
    (1, 1, 3, 5, 0.5, 71),
    (17, 2, 16, 8, 0.4, 72),
    (2, 3, 17, 9, 0.7, 73),
    (1, 5, 33, 16, 0.5, 74),
    (1, 7, 5, 8, 0.3, 75),
]


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
@pytest.mark.parametrize("nC,nA,nV,Q,s,seed", CASES)
def test_energy_and_gradient_at_tile_edges(pk, prec, nC, nA, nV, Q, s, seed):
    p = make_problem(nC, nA, nV, Q, s=s, seed=seed, with_lambda3=True, with_f1=True)
    plan = pk.Plan(nC, nA, nV, Q, precision=prec, grad=True)
    l3, f1 = pk.extra_to_device(p)
    out, dB, de, ds = plan.energy_grad(*pk.to_device(p), p.s, lambda3=l3, f1=f1)
    plan.sync()
    ref = odsrg.energy_and_grad(p.B, p.eps, p.gamma1, p.lambda2, p.s, nC, nA, nV,
                                lambda3=p.lambda3, f1=p.f1)
    dB, de, ds = dB.cpu().numpy(), de.cpu().numpy(), float(ds.cpu()[0])
    errB = np.abs(dB - ref["dB"]).max() / np.abs(ref["dB"]).max()
    erre = np.abs(de - ref["deps"]).max() / np.abs(ref["deps"]).max()
    errs = abs(ds - ref["ds"]) / abs(ref["ds"])
    tol = 1e-10 if prec == "fp64" else 1e-5
    assert errB < tol and erre < tol and errs < tol, (errB, erre, errs)
    if prec == "fp64":
        assert abs(float(out[4].cpu()) - ref["total"]) <= tol * abs(ref["total"])
