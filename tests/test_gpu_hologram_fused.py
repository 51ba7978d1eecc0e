"""The fused steps of the hologram optimisation (csrc/cwo_holo.cu) against the same steps as plain tensor
operators: windows at odd columns, of one row or column, and as large as the canvas."""
import pytest

pytestmark = pytest.mark.gpu
# both sides propagate the same field up to the last bit of its sine and cosine; FP32 propagations
# differ by 3e-7 from the exact ones
TOL = 2e-6


@pytest.fixture(scope="module")
def mods(gpu):
    import torch

    from paper_1107_5578_gb300 import hologram
    return torch, hologram


def _rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


@pytest.mark.parametrize("h,w,canvas", [(96, 160, 256), (33, 77, 128), (1, 64, 64), (64, 1, 64), (128, 128, 128), (255, 511, 512)])
def test_loss_intensity_and_gradient(mods, h, w, canvas):
    torch, hologram = mods
    prob = hologram.HologramProblem(h, w, canvas, 6.4e-6, 520e-9, 0.01)
    g = torch.Generator(device="cuda").manual_seed(h + w)
    phi = (torch.rand((h, w), generator=g, device="cuda") * 6.28).requires_grad_(True)
    geo = hologram._Geometry(prob)
    loss = prob.loss(phi)
    (grad,) = torch.autograd.grad(loss, phi)
    d = geo.intensity(phi) - prob.target
    want = (d * d).mean()
    (wgrad,) = torch.autograd.grad(want, phi)
    assert abs(float(loss) - float(want)) <= TOL * float(want)
    assert _rel(grad, wgrad) <= TOL
    # through the intensity, with a loss of the caller's own and a strided incoming gradient
    wt = torch.rand((w, h), generator=g, device="cuda").t()
    inten = prob.intensity(phi)
    assert _rel(inten.detach(), geo.intensity(phi).detach()) <= TOL
    (grad,) = torch.autograd.grad((inten * wt).sum(), phi)
    (wgrad,) = torch.autograd.grad((geo.intensity(phi) * wt).sum(), phi)
    assert _rel(grad, wgrad) <= TOL
    # a graph of the gradient, a strided phase, and a target changed before the gradient is taken
    (grad2,) = torch.autograd.grad(prob.loss(phi), phi, create_graph=True)
    (wgrad,) = torch.autograd.grad(want_loss(geo, prob, phi), phi)
    assert _rel(grad2.detach(), wgrad) <= TOL
    strided = phi.detach().t().contiguous().t().requires_grad_(True)
    keep = prob.target.clone()
    loss = prob.loss(strided)
    prob.target.zero_()
    loss.backward()
    prob.target.copy_(keep)
    assert _rel(strided.grad, wgrad) <= TOL
    prob.plan.check()


def want_loss(geo, prob, phi):
    d = geo.intensity(phi) - prob.target
    return (d * d).mean()


def test_inputs_the_kernels_do_not_take(mods):
    torch, hologram = mods
    prob = hologram.HologramProblem(20, 30, 64, 6.4e-6, 520e-9, 0.01)
    phi = torch.rand(20, 30, device="cuda", dtype=torch.float64, requires_grad=True)   # composed operators
    loss = prob.loss(phi)
    loss.backward()
    assert phi.grad.dtype == torch.float64
    p32 = phi.detach().float().requires_grad_(True)
    prob.loss(p32).backward()
    assert _rel(p32.grad, phi.grad) <= TOL
    from paper_1107_5578_gb300 import cwo
    x = torch.zeros(64, 64, dtype=torch.complex64, device="cuda")
    image = torch.zeros(20, 30, device="cuda")
    call = cwo.lib().cwo_hologram_forward
    for h, w, ox, oy in ((0, 5, 0, 0), (5, 5, 60, 0), (5, 5, 0, -1), (65, 5, 0, 0)):   # not inside the canvas
        assert call(prob.plan.handle, p32.data_ptr(), None, h, w, ox, oy, x.data_ptr(), image.data_ptr(), None, None, 0) \
            == cwo.ERR_INVALID_ARG
    short = torch.zeros(16, device="cuda")
    big = cwo.Plan(2048, 2048)
    assert call(big.handle, p32.data_ptr(), None, 20, 30, 0, 0, short.data_ptr(), image.data_ptr(), None, None, 0) == cwo.ERR_INVALID_ARG
    # a plan without row windows (a Fresnel one) propagates the whole canvas
    prob.plan = cwo.Plan(64, 64, 6.4e-6, 6.4e-6, 520e-9, 0.01, cwo.FRESNEL_CONV)
    assert prob.plan.rows_group == 0
    geo = hologram._Geometry(prob)
    (grad,) = torch.autograd.grad(prob.loss(p32), p32)
    (want,) = torch.autograd.grad(want_loss(geo, prob, p32), p32)
    assert _rel(grad, want) <= TOL
