"""Batches whose transfer function is evaluated once per call: around the smallest batch that takes that path,
against the same fields one at a time and the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1107_5578_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,b", [(1024, 1024, 7), (1024, 1024, 8), (1024, 512, 7), (1024, 512, 8), (16, 1024, 255), (16, 1024, 256), (512, 512, 17)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_batch_equals_single_calls(gpu, nx, ny, b, adjoint):
    import torch
    from paper_1107_5578_gb300 import cwo
    g = torch.Generator(device="cuda").manual_seed(b)
    x = torch.view_as_complex(torch.randn((b, ny, nx, 2), generator=g, device="cuda"))
    u = synth.random_field(nx, seed=b, ny=ny).astype(np.complex64)
    x[b - 1] = torch.from_numpy(u).cuda()
    plan, other = (cwo.Plan(nx, ny, 8e-6, 6e-6, 532e-9, 0.06) for _ in range(2))
    y = plan.propagate_batch(x, adjoint=adjoint)
    other.propagate_batch(x, z=[0.1] * b)             # per-item distances keep their own evaluation
    z = other.propagate_batch(x, adjoint=adjoint)
    for k in (0, b // 2, b - 1):
        one = plan.adjoint(x[k]) if adjoint else plan.propagate(x[k])
        # the same function evaluated in another kernel: at most a rounding of its phase apart
        assert float((y[k] - one).norm() / one.norm()) <= 1e-6
        assert torch.equal(y[k], z[k])
    want = oracle.propagate(u, 8e-6, 6e-6, 532e-9, 0.06, oracle.ANGULAR, oracle.ADJOINT if adjoint else 0)
    assert np.linalg.norm(y[b - 1].cpu().numpy() - want) / np.linalg.norm(want) <= 2e-5
    plan.check()
