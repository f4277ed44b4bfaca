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


def _gradient_errors(plan, pk, p):
    l3, f1 = pk.extra_to_device(p)
    out, dB, de, ds = plan.energy_grad(*pk.to_device(p), p.s, lambda3=l3, f1=f1)
    plan.sync()
    ref = odsrg.energy_and_grad(p.B, p.eps, p.gamma1, p.lambda2, p.s, p.ncore, p.nactive, p.nvirt,
                                lambda3=p.lambda3, f1=p.f1)
    worst = abs(float(out[4].cpu()) / ref["total"] - 1.0)
    for got, want in ((dB, ref["dB"]), (de, ref["deps"]), (ds, np.asarray([ref["ds"]]))):
        worst = max(worst, np.abs(got.cpu().numpy() - want).max() / np.abs(want).max())
    return worst


def test_workspace_that_cannot_be_allocated(pk, monkeypatch):
    """Only what the CUDA-core kernels need as well may make a plan fail: where the digits'
    workspace cannot be had, the plan runs without it."""
    from paper_1603_00561_gb300 import _native
    sizes = (6, 2, 70, 40)
    p = make_problem(*sizes, s=0.5, seed=5)
    full = pk.Plan(*sizes, precision="fp64", grad=True)
    assert _gradient_errors(full, pk, p) <= 1e-10
    made, smallest = 0, None
    for k in range(80):
        monkeypatch.setenv("DSRG_FAIL_ALLOC_AFTER", str(k))
        try:
            plan = pk.Plan(*sizes, precision="fp64", grad=True)
        except pk.DSRGError as e:
            assert e.status == _native.ERR_OOM and made == 0
            continue
        made += 1
        smallest = plan.workspace_bytes() if smallest is None else smallest
        assert _gradient_errors(plan, pk, p) <= 1e-10
        if plan.workspace_bytes() == full.workspace_bytes():
            break
    assert made > 1 and smallest < full.workspace_bytes()


def _leave_free(torch, nbytes):
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - nbytes, dtype=torch.uint8, device="cuda")


def test_little_free_memory(pk):
    """A plan on a GPU that others have filled takes at most 2/5 of what is left, or does without."""
    import torch
    sizes = (8, 2, 600, 2400)
    p = make_problem(*sizes, s=0.5, seed=6)
    dev = pk.to_device(p)
    plan = pk.Plan(*sizes, precision="fp64")
    ref, need = plan.energy(*dev, p.s).cpu().numpy(), plan.workspace_bytes()
    plan.close()
    filler = _leave_free(torch, 300 << 20)
    try:
        plan = pk.Plan(*sizes, precision="fp64")
        assert plan.workspace_bytes() <= (300 << 20) * 0.5 < need
        e = plan.energy(*dev, p.s).cpu().numpy()
        plan.sync()
        plan.close()
    finally:
        del filler
        torch.cuda.empty_cache()
    assert np.abs(e / ref - 1.0).max() <= 1e-12


def test_batch_under_little_free_memory(pk):
    """The molecules of an FP64 batch share 2/5 of the free memory: those that find no room for
    digits run without. The same energies as plans by themselves."""
    import torch
    sizes = [(8, 2, 300, 1500)] * 5 + [(3, 1, 40, 60)]
    ps = [make_problem(*sz, s=0.5, seed=k) for k, sz in enumerate(sizes)]
    dev = [pk.to_device(p) for p in ps]
    ref = []
    for sz, d, p in zip(sizes, dev, ps):
        plan = pk.Plan(*sz, precision="fp64")
        ref.append(plan.energy(*d, p.s).cpu().numpy())
        plan.close()
    filler = _leave_free(torch, 500 << 20)
    try:
        free0, _ = torch.cuda.mem_get_info()
        batch = pk.Batch(sizes, precision="fp64")
        free1, _ = torch.cuda.mem_get_info()
        e = batch.energy(dev, [p.s for p in ps]).cpu().numpy()
        batch.sync()
        batch.close()
    finally:
        del filler
        torch.cuda.empty_cache()
    # 300 MB or so would not have been left by five digits' workspaces of over 130 MB
    assert free1 >= 0.5 * free0
    assert np.abs(e / np.array(ref) - 1.0).max() <= 1e-12


@pytest.mark.parametrize("world", [20, 21, 22, 1000, 30_000_000, 100_000_000, 2 ** 31 - 1])
def test_shards_of_a_world_with_more_ranks_than_pairs(pk, world):
    """21 core pairs: from 21 ranks on a rank has one pair or none, however many there are."""
    nC = 6
    p = make_problem(nC, 0, 70, 40, s=0.5, seed=8)
    dev = pk.to_device(p)
    plan = pk.Plan(nC, 0, 70, 40, precision="fp64")
    pairs = plan.pair_energies(dev[0], dev[1], p.s).cpu().numpy()
    iu = [(i, j) for i in range(nC) for j in range(i, nC)]
    for rank in (0, 3, 19, 20, world - 1):
        if rank >= world:
            continue
        plan.set_shard(rank, world)
        e = plan.energy(*dev, p.s).cpu().numpy()
        plan.sync()
        want = sum((1.0 if i == j else 2.0) * pairs[i, j] for k, (i, j) in enumerate(iu) if k % world == rank)
        assert abs(e[0] - want) <= 1e-12 * abs(pairs).sum()


@pytest.mark.parametrize("sizes", [(1, 1, 3, 5), (3, 3, 33, 20), (2, 5, 17, 9), (2, 8, 40, 30), (5, 0, 65, 17)])
def test_plan_without_digits(pk, monkeypatch, sizes):
    """The CUDA-core kernels for every kind of active space, with the inputs of the full Table 1:
    the plan of the first allocation count that suffices."""
    p = make_problem(*sizes, s=0.6, seed=11, with_lambda3=sizes[1] > 0, with_f1=True)
    for k in range(80):
        monkeypatch.setenv("DSRG_FAIL_ALLOC_AFTER", str(k))
        try:
            plan = pk.Plan(*sizes, precision="fp64", grad=True)
            break
        except pk.DSRGError:
            continue
    monkeypatch.delenv("DSRG_FAIL_ALLOC_AFTER")
    full = pk.Plan(*sizes, precision="fp64", grad=True)
    assert plan.workspace_bytes() < full.workspace_bytes()
    assert _gradient_errors(plan, pk, p) <= 1e-10
    assert _gradient_errors(full, pk, p) <= 1e-10
