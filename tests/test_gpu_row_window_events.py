"""Timing events of a plan are recorded by every call that propagates, row windows and hologram steps included."""
import pytest

pytestmark = pytest.mark.gpu


def _events(torch):
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
    for e in ev:
        e.record()
    return ev


@pytest.mark.parametrize("nx,ny,cached", [(256, 256, False), (512, 128, True), (4096, 64, False)])
def test_row_windows_record(gpu, nx, ny, cached):
    import torch
    from paper_1107_5578_gb300 import cwo
    plan = cwo.Plan(nx, ny, 8e-6, 6e-6, 532e-9, 0.03, cwo.ANGULAR, cwo.FLAG_CACHE_H if cached else 0)
    x = torch.zeros(ny, nx, dtype=torch.complex64, device="cuda")
    ev = _events(torch)
    plan.set_timing_events(ev)
    for adjoint in (False, True):
        mark = torch.cuda.Event(enable_timing=True)
        mark.record()
        plan.propagate_rows(x, (8, 16), (0, 8), adjoint=adjoint)
        torch.cuda.synchronize()
        assert mark.elapsed_time(ev[0]) >= 0.0        # recorded by this call
        assert all(a.elapsed_time(b) > 0.0 for a, b in zip(ev, ev[1:]))
    plan.set_timing_events(None)
    plan.check()


def test_hologram_step_records(gpu):
    import torch
    from paper_1107_5578_gb300 import hologram
    prob = hologram.HologramProblem(30, 40, 64, 6.4e-6, 520e-9, 0.01)
    phi = torch.zeros(30, 40, device="cuda", requires_grad=True)
    ev = _events(torch)
    prob.plan.set_timing_events(ev)
    mark = torch.cuda.Event(enable_timing=True)
    mark.record()
    loss = prob.loss(phi)
    torch.cuda.synchronize()
    assert mark.elapsed_time(ev[0]) >= 0.0
    mark.record()
    loss.backward()
    torch.cuda.synchronize()
    assert mark.elapsed_time(ev[0]) >= 0.0 and all(a.elapsed_time(b) > 0.0 for a, b in zip(ev, ev[1:]))
