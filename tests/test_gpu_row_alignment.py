"""Inputs on and off a 16-byte boundary: between padded rows of 512 and 4096 values the forward row pass has a kernel
of bulk copies for the first and one of per-thread loads for the second, outside them one kernel for both."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(128, 64), (256, 64), (512, 32), (2048, 64), (4096, 64)])
def test_input_off_a_16_byte_boundary(gpu, nx, ny):
    import torch
    from paper_1107_5578_gb300 import cwo
    plan = cwo.Plan(nx, ny, 8e-6, 6e-6, 532e-9, 0.03)
    g = torch.Generator(device="cuda").manual_seed(nx)
    x = torch.view_as_complex(torch.randn((ny, nx, 2), generator=g, device="cuda"))
    buf = torch.empty(nx * ny + 1, dtype=torch.complex64, device="cuda")
    off = buf[1:].view(ny, nx)
    off.copy_(x)
    assert x.data_ptr() % 16 == 0 and off.data_ptr() % 16 == 8
    a, b = plan.propagate(x), plan.propagate(off)
    # the same transforms of the same values in the same order
    assert float((a - b).norm()) <= 1e-6 * float(a.norm())
    plan.check()
