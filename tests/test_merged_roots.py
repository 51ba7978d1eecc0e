"""The 16-point DFT with merged roots (padded length 4096; 2048 in shifted plans, 8192 in split rows) against the oracle.  Bounds: a padded 4096-point
transform pair rounds each value about 2 x 12 levels at 6e-8, rms about 6e-8 sqrt(24) = 3e-7 an axis; with
the tables' 1e-7 a value under 1e-6, and four times that is allowed."""
import numpy as np
import pytest

import oracle
from paper_1107_5578_gb300 import cwo, synth

TOL = 4e-6


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("nx,ny", [(16, 2048), (2048, 16)])
@pytest.mark.parametrize("kind,z", [(0, 0.02), (1, 0.05)])
@pytest.mark.parametrize("adjoint", [0, 1])
def test_emulated_axis_of_4096(nx, ny, kind, z, adjoint):
    u = synth.random_field(nx, seed=nx + kind, ny=ny)
    got = cwo.emulate(u.astype(np.complex64), 8e-6, 8e-6, 532e-9, z, kind, 0, adjoint)
    assert rel(got, oracle.propagate(u, 8e-6, 8e-6, 532e-9, z, kind, oracle.ADJOINT if adjoint else 0)) <= TOL


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(16, 2048), (2048, 32), (512, 2048), (2048, 512), (32, 1024), (4096, 1024)])
@pytest.mark.parametrize("form", ["asm", "cached", "fresnel", "shifted", "stack"])
def test_axis_of_4096(gpu, nx, ny, form):
    import torch
    batch, z = 3, 0.03
    u = np.stack([synth.random_field(nx, seed=nx + ny + k, ny=ny) for k in range(batch)])
    x = torch.from_numpy(u.astype(np.complex64)).cuda()
    kind = cwo.FRESNEL_CONV if form in ("fresnel", "stack") else cwo.ANGULAR
    kw, zs, want = {}, [z] * batch, lambda k: oracle.propagate(u[k], 8e-6, 8e-6, 532e-9, z, kind)
    if form == "cached":
        kw["flags"] = cwo.FLAG_CACHE_H
    elif form == "shifted":
        kw["shift"] = cwo.Shift(2e-4, -1e-4, 0.0, 0.0, 0.0, 0.0)
        want = lambda k: oracle.propagate_shifted(u[k], 8e-6, 8e-6, 532e-9, z, 2e-4, -1e-4, 0.0, 0.0, 0.0, 0.0)
    if form == "stack":
        zs = [0.03, 0.05, -0.04]
        want = lambda k: oracle.propagate(u[0], 8e-6, 8e-6, 532e-9, zs[k], cwo.FRESNEL_CONV)
    plan = cwo.Plan(nx, ny, 8e-6, 8e-6, 532e-9, z, kind, **kw)
    y = (plan.propagate_stack(x[0].contiguous(), zs) if form == "stack" else plan.propagate_batch(x)).cpu().numpy()
    plan.check()
    plan.close()
    for k in range(batch):
        assert rel(y[k], want(k)) <= TOL
