"""Per-item angular-spectrum tables formed on the device: batches around the number of items of one table
launch, bit for bit what a single call computes."""
import numpy as np
import pytest

import oracle
from paper_1107_5578_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cwo(gpu):
    import paper_1107_5578_gb300.cwo as m
    m.lib()
    return m


@pytest.mark.parametrize("nx,ny,b", [(16, 16, 1), (64, 32, 24), (32, 64, 25), (16, 128, 49), (2048, 16, 3)])
def test_distances_equal_to_the_plans_own(cwo, nx, ny, b):
    # the plan's tables come from the host, the per-distance ones from the device: the same bits
    import torch
    x = torch.from_numpy(np.stack([synth.random_field(nx, seed=k, ny=ny) for k in range(b)]).astype(np.complex64)).cuda()
    for z in (0.07, -0.013):
        plan = cwo.Plan(nx, ny, 8e-6, 6e-6, 532e-9, z)
        y = plan.propagate_batch(x, z=[z] * b)
        assert torch.equal(y, plan.propagate_batch(x))
        plan.check()


@pytest.mark.parametrize("nx,ny,b", [(32, 16, 24), (16, 64, 25), (64, 64, 50)])
def test_items_around_one_table_launch(cwo, nx, ny, b):
    # angular-spectrum and Fresnel items in runs of changing length; every item as if alone
    import torch
    x = torch.from_numpy(np.stack([synth.random_field(nx, seed=k, ny=ny) for k in range(b)]).astype(np.complex64)).cuda()
    items = [dict(type=int(k % 7 in (2, 3, 6)), z=0.004 + 0.003 * k, wavelength=(450e-9, 532e-9, 633e-9)[k % 3],
                  dx=5e-6 + 1e-7 * k, dy=6e-6) for k in range(b)]
    plan = cwo.Plan(nx, ny)
    y = plan.propagate_items(x, items)
    off = torch.empty(b * nx * ny + 1, dtype=torch.complex64, device="cuda")[1:].view(b, ny, nx)   # off 16 bytes: three passes
    plan.propagate_items(x, items, out=off)
    plan.check()
    for k in (0, 2, 22, 23, b - 1):
        assert torch.equal(plan.propagate_items(x[k:k + 1], items[k:k + 1])[0], y[k]), k
        it = items[k]
        want = oracle.propagate(x[k].cpu().numpy(), it["dx"], it["dy"], it["wavelength"], it["z"], it["type"])
        for got in (y[k], off[k]):
            assert np.linalg.norm(got.cpu().numpy() - want) / np.linalg.norm(want) <= 2e-5, k
