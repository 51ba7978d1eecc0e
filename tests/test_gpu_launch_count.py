"""Launches of a batched call: what Plan.launches_per_batch says against the kernels that a stream capture of the
call holds."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu
KERNEL = 0   # CU_GRAPH_NODE_TYPE_KERNEL


def _kernels(torch, call):
    """number of kernel nodes that `call(stream)` captures"""
    cu = ctypes.CDLL("libcuda.so.1")
    s = torch.cuda.Stream()
    h, graph, n = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(h, 2) == 0          # relaxed
    call(s)
    assert cu.cuStreamEndCapture(h, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    count = 0
    for node in nodes:
        kind = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        count += kind.value == KERNEL
    cu.cuGraphDestroy(graph)
    return count


# one field; a large batch of small fields and the batch below it; per-item distances in two table launches and in
# FP64 per element; the Fresnel form
@pytest.mark.parametrize("n,b,kind,pitch,z", [
    (512, 1, 0, 8e-6, None), (512, 15, 0, 8e-6, None), (512, 16, 0, 8e-6, None), (64, 30, 0, 8e-6, 0.05),
    (64, 3, 0, 1e-6, 0.05), (512, 16, 1, 8e-6, None)])
def test_launches(gpu, n, b, kind, pitch, z):
    import torch
    from paper_1107_5578_gb300 import cwo
    plan = cwo.Plan(n, n, pitch, pitch, 532e-9, 0.05, kind)
    plan.reserve(b)
    x = torch.zeros(b, n, n, dtype=torch.complex64, device="cuda")
    out = torch.empty_like(x)
    zs = None if z is None else [z * (1 + 0.01 * k) for k in range(b)]
    if zs is not None:
        plan.propagate_batch(x, z=[0.7 * v for v in zs])     # per-item tables of other distances: allocated
    torch.cuda.synchronize()
    want = plan.launches_per_batch(b, zs)
    assert _kernels(torch, lambda s: plan.propagate_batch(x, z=zs, out=out, stream=s)) == want
    if b == 1:
        assert want == plan.launches_per_call
    torch.cuda.synchronize()
