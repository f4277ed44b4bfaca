"""The FP64 products on the tensor cores (csrc/oz_gemm.cu) through FP64 plans.

The digits of constant factors are all at their largest, so the integer sums of
the tensor cores come as near 2^24 as they can; K and the virtual space run over
the edges of the kernel's stages (32), chunks (128) and tiles (64, 128). Bar:
pair energies are sums of positive terms v^2 R with v off by at most one rounding
(2^-53) plus the slicing (2^-56 of the largest value, here the value itself), R by
a few roundings, so 16 x 2^-52 relative holds them (energies of mixed signs: the
1e-10 bar of the FP64 tests).
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


# digits 127 ... and -128 ... (base 256, value below 1): the largest same-sign products
TOP = sum(127.0 * 256.0 ** -i * 2.0 for i in range(1, 8))


@pytest.mark.parametrize("x", [TOP, -TOP, 1.0, 0.75 * 2.0 ** -400, 3.0 ** 20])
@pytest.mark.parametrize("Q,nV", [(1, 3), (31, 63), (32, 64), (33, 65), (128, 128), (129, 130), (900, 40)])
def test_constant_factors(pk, x, Q, nV):
    import torch
    p = make_problem(2, 0, nV, Q, s=0.5, seed=1)
    B = torch.full((Q, 2, nV), x, dtype=torch.float64, device="cuda")
    eps = torch.as_tensor(p.eps).cuda()
    plan = pk.Plan(2, 0, nV, Q, precision="fp64")
    e = plan.pair_energies(B, eps, 0.5).cpu().numpy()
    plan.sync()
    v = np.longdouble(x) ** 2 * Q
    eC, eV = p.eps[:2].astype(np.longdouble), p.eps[2:].astype(np.longdouble)
    for i in range(2):
        for j in range(2):
            D = eC[i] + eC[j] - eV[:, None] - eV[None, :]
            ref = np.sum(v * v * -np.expm1(-2 * np.longdouble(0.5) * D * D) / D)
            if abs(ref) > 1e-300:
                assert abs(e[i, j] / ref - 1) <= 16 * 2.0 ** -52, (i, j, e[i, j], ref)


@pytest.mark.parametrize("nC,nA,nV,Q,seed", [(3, 1, 5, 7, 0), (2, 8, 33, 40, 1), (5, 3, 129, 161, 2),
                                             (4, 2, 200, 300, 3)])
def test_wide_ranges(pk, nC, nA, nV, Q, seed):
    """Rows of very different sizes, and values within a row over 60 binary orders."""
    p = make_problem(nC, nA, nV, Q, s=0.7, seed=seed, b_decay=0.0)
    r = np.random.default_rng(seed)
    B = p.B * 2.0 ** r.integers(-30, 30, p.B.shape)
    B[:, nC:, :nA] = 0.5 * (B[:, nC:, :nA] + B[:, nC:, :nA].transpose(0, 2, 1))
    ref = odsrg.energy(B, p.eps, p.gamma1, p.lambda2, p.s, nC, nA, nV)
    import torch
    q = type(p)(**{**p.__dict__, "B": B})
    plan = pk.Plan(nC, nA, nV, Q, precision="fp64")
    out = plan.energy(*pk.to_device(q), p.s).cpu().numpy()
    plan.sync()
    for k, v in zip(pk.BLOCKS, out):
        assert abs(v - ref[k]) <= 1e-10 * abs(ref[k]), (k, v, ref[k])


def test_not_finite(pk):
    """A NaN row gives NaN; an infinite factor that meets only zeros elsewhere in its
    products gives NaN (inf * 0) as in FP64, one that meets finite values +-inf or NaN."""
    import torch
    p = make_problem(3, 2, 70, 40, s=0.5, seed=4)
    B, eps, g, l = pk.to_device(p)
    plan = pk.Plan(3, 2, 70, 40, precision="fp64")
    good = plan.energy(B, eps, g, l, p.s).clone()
    for bad in (float("nan"), float("inf")):
        Bb = B.clone()
        Bb[5, 1, 30] = bad
        e = plan.pair_energies(Bb, eps, p.s).cpu().numpy()
        fine = np.ones((3, 3), dtype=bool)
        fine[1, :] = fine[:, 1] = False
        ok = plan.pair_energies(B, eps, p.s).cpu().numpy()
        assert not np.isfinite(e[~fine]).any()
        assert np.array_equal(e[fine], ok[fine])
    assert torch.equal(plan.energy(B, eps, g, l, p.s), good)
    plan.sync()
