"""dsrg_plan_last_launch_count against the kernel nodes of the captured call."""
import ctypes as C

import pytest

from dsrg_synth import make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1603_00561_gb300 as pk
    pk.build()
    return pk


def _kernel_nodes(stream, call):
    """Kernel nodes of the graph that the driver captures from `call` on `stream`."""
    cu = C.CDLL("libcuda.so.1")
    s, graph = C.c_void_p(stream.cuda_stream), C.c_void_p()
    assert cu.cuStreamBeginCapture_v2(s, 2) == 0  # relaxed
    try:
        call()
    finally:
        assert cu.cuStreamEndCapture(s, C.byref(graph)) == 0
    n = C.c_size_t()
    assert cu.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, C.byref(n)) == 0
    kernels = 0
    for k in range(n.value):
        kind = C.c_int()
        assert cu.cuGraphNodeGetType(C.c_void_p(nodes[k]), C.byref(kind)) == 0
        kernels += kind.value == 0
    assert cu.cuGraphDestroy(graph) == 0
    return kernels


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
@pytest.mark.parametrize("sizes", [(6, 2, 150, 90), (3, 0, 40, 30), (4, 5, 60, 50)])
def test_launch_count(pk, prec, sizes):
    import torch
    p = make_problem(*sizes, s=0.5, seed=9)
    plan = pk.Plan(*sizes, precision=prec, grad=True)
    dev = pk.to_device(p)
    out = torch.zeros(5, dtype=torch.float64, device="cuda")
    dB, de = torch.zeros_like(dev[0]), torch.zeros_like(dev[1])
    ds = torch.zeros(1, dtype=torch.float64, device="cuda")
    ptr = lambda t: None if t is None else C.c_void_p(t.data_ptr())
    args = [plan.h] + [ptr(t) for t in dev] + [p.s, ptr(out)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        plan.energy_grad(*dev, p.s)  # sets the plan's stream
        torch.cuda.synchronize()
        for call in (lambda: plan.lib.dsrg_mrpt2_energy(*args),
                     lambda: plan.lib.dsrg_mrpt2_energy_grad(*args, ptr(dB), ptr(de), ptr(ds))):
            n = _kernel_nodes(stream, lambda: call() == 0 or pytest.fail("the call failed"))
            assert plan.last_launch_count() == n
    plan.close()
