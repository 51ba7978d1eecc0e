"""Hologram gradients under saved-tensor hooks that hand the saved tensors back in another type, stride or shape."""
import pytest

pytestmark = pytest.mark.gpu


def _grad(prob, phi, unpack, through_intensity):
    import torch
    with torch.autograd.graph.saved_tensors_hooks(lambda t: t, unpack):
        loss = prob.intensity(phi).sum() if through_intensity else prob.loss(phi)
    return torch.autograd.grad(loss, phi)[0]


@pytest.mark.parametrize("through_intensity", [False, True])
def test_gradient_under_hooks(gpu, through_intensity):
    import torch
    from paper_1107_5578_gb300 import hologram
    prob = hologram.HologramProblem(20, 30, 64, 6.4e-6, 520e-9, 0.01)
    phi = torch.rand(20, 30, device="cuda", requires_grad=True)
    want = _grad(prob, phi, lambda t: t, through_intensity)
    wide = {torch.float32: torch.float64, torch.complex64: torch.complex128}
    assert torch.equal(_grad(prob, phi, lambda t: t.to(wide[t.dtype]), through_intensity), want)
    assert torch.equal(_grad(prob, phi, lambda t: t.t().contiguous().t(), through_intensity), want)
    with pytest.raises(RuntimeError):
        _grad(prob, phi, lambda t: t.t().contiguous(), through_intensity)
    prob.plan.check()
