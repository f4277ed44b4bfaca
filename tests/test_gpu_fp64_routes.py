"""FP64 plans by both of their routes: the digit products on the tensor cores
(csrc/fp64_tc.cu) and the CUDA-core kernels, which take over where the digits' workspace
does not fit. Bar: 1e-10 relative, the FP64 bar of the other tests.
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


@pytest.mark.parametrize("naux", [(1 << 21) - 1, (1 << 21) + 1, 5_000_000])
def test_very_long_auxiliary_basis(pk, naux):
    """naux around the limit of the digit products, and past the 65535 blocks of 64 that one grid
    dimension has."""
    import torch
    plan = pk.Plan(1, 0, 1, naux, precision="fp64")
    B = torch.randn((naux, 1, 1), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(1))
    eps = torch.tensor([-1.0, 0.5], dtype=torch.float64, device="cuda")
    e = plan.energy(B, eps, None, None, 0.5).cpu().numpy()
    plan.sync()
    v = float((B * B).sum())
    ref = v * v * -np.expm1(-9.0) / -3.0
    assert abs(e[4] / ref - 1.0) <= 1e-10
