"""Hologram step on the largest canvas: the plan has no cached transfer function there, so that the row windows run
the split row passes and the column kernel that evaluates H."""
import pytest

pytestmark = pytest.mark.gpu
TOL = 2e-6   # as for the smaller canvases: the same propagation up to the last bit of a sine


@pytest.mark.parametrize("h,w", [(2160, 3840), (1, 4096), (4096, 7)])
def test_step_on_the_largest_canvas(gpu, h, w):
    import torch
    from paper_1107_5578_gb300 import cwo, hologram
    prob = hologram.HologramProblem(h, w, 4096, 3.74e-6, 520e-9, 0.05)
    assert prob.plan.flags & cwo.FLAG_CACHE_H == 0 and prob.plan.rows_group > 0
    g = torch.Generator(device="cuda").manual_seed(h)
    phi = (torch.rand((h, w), generator=g, device="cuda") * 6.28).requires_grad_(True)
    loss = prob.loss(phi)
    (grad,) = torch.autograd.grad(loss, phi)
    d = hologram._Geometry(prob).intensity(phi) - prob.target
    want = (d * d).mean()
    (wgrad,) = torch.autograd.grad(want, phi)
    assert abs(float(loss.detach()) - float(want.detach())) <= TOL * float(want.detach())
    assert float((grad.double() - wgrad.double()).norm()) <= TOL * float(wgrad.double().norm())
    prob.plan.check()
