"""A field's result does not depend on the batch it rides in, bit for bit: mixed batches of 1024-row items, and
batches at the plan's distance on both sides of the size from which the transfer function is evaluated once per
call; with the remainder of the phase as a series and in closed form."""
import pytest

pytestmark = pytest.mark.gpu
# (pitch, z): remainder as a series / in closed form
TAILS = {"series": (8e-6, 0.06), "closed": (1e-6, 5e-4)}


def _fields(b, ny, nx):
    import torch
    g = torch.Generator(device="cuda").manual_seed(b + ny)
    return torch.view_as_complex(torch.randn((b, ny, nx, 2), generator=g, device="cuda"))


@pytest.mark.parametrize("nx,ny", [(1024, 1024), (64, 1024), (512, 512)])
def test_items_alone_and_together(gpu, nx, ny):
    import torch
    from paper_1107_5578_gb300 import cwo
    # FP64 phases (a far plane of fine pitch) and a Fresnel item among them
    geo = [(0, 8e-6, 0.06), (0, 1e-6, 5e-4), (0, 1e-6, 0.05), (0, 4e-6, 0.3), (0, 1e-6, 2e-4), (0, 8e-6, -0.1), (1, 8e-6, 0.2), (0, 6e-6, 0.01)]
    items = [{"type": k, "z": z, "wavelength": 532e-9, "dx": p} for k, p, z in geo]
    x = _fields(len(items), ny, nx)
    plan = cwo.Plan(nx, ny)
    alone = [plan.propagate_items(x[k:k + 1], [items[k]])[0] for k in range(len(items))]
    for lo, hi in ((0, 2), (0, 4), (1, 6), (0, 8)):
        y = plan.propagate_items(x[lo:hi].contiguous(), items[lo:hi])
        for k in range(lo, hi):
            assert torch.equal(y[k - lo], alone[k]), (lo, hi, k)
    plan.check()


@pytest.mark.parametrize("tail", TAILS)
@pytest.mark.parametrize("nx,ny,b", [(1024, 1024, 5), (1024, 1024, 8), (1024, 512, 8), (512, 512, 17), (16, 1024, 256), (1024, 16, 256)])
def test_batch_equals_single_calls_bit_for_bit(gpu, nx, ny, b, tail):
    import torch
    from paper_1107_5578_gb300 import cwo
    pitch, z = TAILS[tail]
    plan = cwo.Plan(nx, ny, pitch, pitch, 532e-9, z)
    x = _fields(b, ny, nx)
    for adjoint in (False, True):
        y = plan.propagate_batch(x, adjoint=adjoint)
        i = plan.propagate_epilogue(x, cwo.EPI_INTENSITY, adjoint=adjoint)
        zs = plan.propagate_batch(x, z=[z] * b, adjoint=adjoint)
        for k in (0, b // 2, b - 1):
            one = plan.adjoint(x[k]) if adjoint else plan.propagate(x[k])
            assert torch.equal(y[k], one), (adjoint, k)
            assert torch.equal(zs[k], one), (adjoint, k)
            assert torch.equal(i[k], plan.propagate_epilogue(x[k], cwo.EPI_INTENSITY, adjoint=adjoint)), (adjoint, k)
    plan.check()


def test_gs_batch_equals_single_runs(gpu):
    import torch
    from paper_1107_5578_gb300 import cwo
    n, b = 512, 17
    plan = cwo.Plan(n, n, 8e-6, 8e-6, 532e-9, 0.06)
    f = _fields(b, n, n)
    amp = f.abs().contiguous()
    whole = f.clone()
    inten = plan.gs_run(amp, whole, 1)
    for k in (0, b - 1):
        one = f[k].clone()
        i = plan.gs_run(amp[k].contiguous(), one, 1)
        assert torch.equal(one, whole[k]) and torch.equal(i.view(n, n), inten[k])
    plan.check()
