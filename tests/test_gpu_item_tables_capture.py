"""Per-item distances under stream capture: the tables of a captured call are formed when the graph runs, not when
it is captured, so no later call may take them as made, and a replay may not leave another call's in use."""
import pytest

pytestmark = pytest.mark.gpu


def test_captured_distances(gpu):
    import torch
    from paper_1107_5578_gb300 import cwo
    n, b = 128, 3
    za, zb, zc = ([z * (1 + 0.1 * k) for k in range(b)] for z in (0.02, 0.05, 0.09))
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.view_as_complex(torch.randn((b, n, n, 2), generator=g, device="cuda"))
    want = {id(z): cwo.Plan(n, n, 8e-6, 8e-6, 532e-9, 0.05).propagate_batch(x, z=z) for z in (za, zb, zc)}
    plan = cwo.Plan(n, n, 8e-6, 8e-6, 532e-9, 0.05)
    plan.reserve(b)
    assert torch.equal(plan.propagate_batch(x, z=za), want[id(za)])
    out, out2 = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    graph, graph2 = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.propagate_batch(x, z=zb, out=out)
    with torch.cuda.graph(graph2):                                        # the distances of an earlier eager call
        plan.propagate_batch(x, z=za, out=out2)
    assert torch.equal(plan.propagate_batch(x, z=zb), want[id(zb)])       # before any replay
    assert torch.equal(plan.propagate_batch(x, z=zc), want[id(zc)])
    graph.replay()
    assert torch.equal(out, want[id(zb)])
    assert torch.equal(plan.propagate_batch(x, z=zc), want[id(zc)])       # after it
    graph2.replay()
    assert torch.equal(out2, want[id(za)])
    plan.check()
