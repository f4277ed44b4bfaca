"""A NaN in any input array comes out of the energy as NaN, in every precision: also where
minima and maxima that skip NaNs choose the path of the regulators."""
import numpy as np
import pytest

from dsrg_synth import make_problem

pytestmark = pytest.mark.gpu

SIZES = (5, 2, 150, 70)
nC, nA, nV, Q = SIZES


@pytest.fixture(scope="module")
def pk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1603_00561_gb300 as pk
    pk.build()
    return pk


WHERE = [
    # array, element, blocks that read it (by BLOCKS' index)
    ("B", (3, 1, nA + 7), (0, 1, 2)), ("B", (3, nC + 1, nA + 7), (1, 3)), ("B", (40, 2, nA + 149), (0, 1, 2)),
    ("B", (69, nC, 1), (3,)),
    ("eps", (0,), (0, 1, 2)), ("eps", (nC,), (1, 2, 3)), ("eps", (nC + nA,), (0, 1, 2, 3)),
    ("eps", (nC + nA + 127,), (0, 1, 2, 3)), ("eps", (nC + nA + 149,), (0, 1, 2, 3)),
    ("gamma1", (0, 1), (1, 2, 3)), ("lambda2", (0, 1, 1, 0), (3,)),
    ("lambda3", (0, 1, 2, 0, 1, 2), (3,)), ("f1", (1, nA + 3), (3,)),
]


@pytest.mark.parametrize("prec", ["fp64", "bf16x3", "tf32x3"])
@pytest.mark.parametrize("name,at,blocks", WHERE)
def test_nan_propagates(pk, prec, name, at, blocks):
    p = make_problem(*SIZES, s=0.5, seed=21, with_lambda3=True, with_f1=True)
    B, eps, G, L = pk.to_device(p)
    l3, f1 = pk.extra_to_device(p)
    dict(B=B, eps=eps, gamma1=G, lambda2=L, lambda3=l3, f1=f1)[name][at] = float("nan")
    plan = pk.Plan(*SIZES, precision=prec)
    e = plan.energy(B, eps, G, L, p.s, lambda3=l3, f1=f1).cpu().numpy()
    plan.sync()
    assert np.isnan(e[4])
    assert np.isnan(e[list(blocks)]).all(), e
