"""Device memory of a plan: cwo_plan_device_bytes grows by the same amount with every field, and cwo_plan_reserve
holds the tables and the fields' scratch and nothing else."""
import pytest

from paper_1107_5578_gb300 import cwo


@pytest.mark.parametrize("nx,ny,b", [(1024, 1024, 8), (512, 512, 16), (16, 1024, 256)])
def test_device_bytes_are_linear_in_the_batch(nx, ny, b):
    d = [cwo.device_bytes(nx, ny, k) for k in (b - 2, b - 1, b, b + 1)]
    assert d[1] - d[0] == d[2] - d[1] == d[3] - d[2]


@pytest.mark.gpu
@pytest.mark.parametrize("batch", [7, 16])
def test_reserve_holds_what_device_bytes_says(gpu, batch):
    import torch
    nx = ny = 1024
    cwo.Plan(nx, ny).propagate(torch.zeros(ny, nx, dtype=torch.complex64, device="cuda"))   # kernels loaded
    torch.cuda.synchronize()
    plan = cwo.Plan(nx, ny)
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    before = cwo.device_bytes(nx, ny, 1)
    plan.reserve(batch)
    held = free - torch.cuda.mem_get_info()[0]
    field = 8 * ny * 2 * nx
    # one field more than asked for (the source of a stack), rounded up to the driver's 2 MB pages
    assert held <= cwo.device_bytes(nx, ny, batch) - before + field + (6 << 20)
