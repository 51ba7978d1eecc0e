"""A HologramProblem whose steps a program has replaced (a subclass with its own field, an instance with its own
intensity) computes its loss through them."""
import pytest

pytestmark = pytest.mark.gpu


def _step(prob, phi):
    import torch
    loss = prob.loss(phi)
    return loss.detach(), torch.autograd.grad(loss, phi)[0], prob.intensity(phi).detach()


def test_replaced_steps_are_used(gpu):
    import torch
    from paper_1107_5578_gb300 import hologram

    class Brighter(hologram.HologramProblem):
        def field(self, phi):
            return 2.0 * super().field(phi)

    class Squared(hologram.HologramProblem):
        def intensity(self, phi):
            return super().intensity(phi) ** 2

    args = (20, 30, 64, 6.4e-6, 520e-9, 0.01)
    phi = torch.rand(20, 30, device="cuda", requires_grad=True)
    plain = hologram.HologramProblem(*args)
    t, inten = plain.target, plain.intensity(phi).detach()
    brighter, squared, instance = Brighter(*args), Squared(*args), hologram.HologramProblem(*args)
    instance.field = brighter.field
    for prob, want in ((brighter, 4.0 * inten), (squared, inten ** 2), (instance, 4.0 * inten)):
        prob.target = t
        loss, grad, got = _step(prob, phi)
        # the same propagation to single precision
        assert float((got - want).norm()) <= 4e-6 * float(want.norm())
        wl = ((want.double() - t.double()) ** 2).mean()
        assert abs(float(loss) - float(wl)) <= 1e-5 * float(wl)
        assert grad.shape == phi.shape and float(grad.norm()) > 0.0
