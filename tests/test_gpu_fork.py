"""An energy call whose blocks run on two streams: nothing of one call may reach into
the next one on the same plan, nor into another plan's on another thread and stream.
The same numbers, bit for bit, as calls with a synchronisation after each.

Sizes: fewer CCVV work items than SMs, and several times more.
"""
import threading

import pytest

from dsrg_synth import make_problem

pytestmark = pytest.mark.gpu

SIZES = [(5, 2, 70, 60), (20, 3, 300, 64)]


@pytest.fixture(scope="module")
def pk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1603_00561_gb300 as pk
    pk.build()
    return pk


def problems(pk, size):
    ps = [make_problem(*size, s=0.5, seed=s) for s in (81, 82)]
    return [(pk.to_device(p), p.s) for p in ps]


@pytest.mark.parametrize("size", SIZES)
def test_calls_in_a_row_and_in_threads(pk, size):
    import torch
    plan = pk.Plan(*size, precision="bf16x3")
    inputs = problems(pk, size)
    ref = []
    for dev, s in inputs:
        ref.append(plan.energy(*dev, s).clone())
        torch.cuda.synchronize()
    # alternating inputs with no synchronisation between the calls
    outs = [plan.energy(*inputs[k % 2][0], inputs[k % 2][1]).clone() for k in range(12)]
    torch.cuda.synchronize()
    assert all(torch.equal(o, ref[k % 2]) for k, o in enumerate(outs))
    plan.sync()
    # a plan, a stream and an input per thread
    got, errors = [None, None], []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                own = pk.Plan(*size, precision="bf16x3")
                got[i] = [own.energy(*inputs[i][0], inputs[i][1]).clone() for _ in range(8)]
                own.sync()
        except Exception as e:  # reported by the assertion below
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    assert all(torch.equal(o, ref[i]) for i in (0, 1) for o in got[i])
