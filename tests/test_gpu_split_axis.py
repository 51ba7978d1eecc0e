"""Axes of 4096 samples (padded to 8192): the split row passes along x, and the tables in their order
beside those of the line and column passes, for every diffraction type, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1107_5578_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 2e-5   # relative L2, the library's bar
SHAPES = [(4096, 16), (4096, 64), (16, 4096), (64, 4096)]
LAM, PITCH = 532e-9, 5e-6


@pytest.fixture(scope="module")
def cwo(gpu):
    import paper_1107_5578_gb300.cwo as m
    m.lib()
    return m


def _fields(nx, ny, b, seed):
    return np.stack([synth.random_field(nx, seed=seed + k, ny=ny) for k in range(b)]).astype(np.complex64)


def _err(got, want):
    return np.linalg.norm(got.cpu().numpy().astype(np.complex128) - want) / np.linalg.norm(want)


def _off16(torch, a):
    """a copy of the batch that starts 8 bytes off a 16-byte boundary"""
    t = torch.empty(a.numel() + 1, dtype=a.dtype, device=a.device)[1:].view(a.shape)
    return t.copy_(a)


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("kind", [0, 1])
def test_batch_adjoint_distances_alignment(cwo, nx, ny, kind):
    import torch
    u = _fields(nx, ny, 3, nx + ny + kind)
    x = torch.from_numpy(u).cuda()
    for flags in ((0, cwo.FLAG_CACHE_H) if kind == 0 else (0, cwo.FLAG_LITERAL_SCALE)):
        plan = cwo.Plan(nx, ny, PITCH, 6e-6, LAM, 0.08, kind, flags)
        of = oracle.LITERAL_SCALE if flags == cwo.FLAG_LITERAL_SCALE else 0
        y, ya = plan.propagate_batch(x), plan.propagate_batch(x, adjoint=True)
        yo = plan.propagate_batch(_off16(torch, x), out=_off16(torch, x))   # Fresnel: three passes
        yz = plan.propagate_batch(x, z=[0.05, 0.08, 0.11])
        plan.check()
        for k in range(3):
            want = oracle.propagate(u[k], PITCH, 6e-6, LAM, 0.08, kind, of)
            assert _err(y[k], want) <= TOL and _err(yo[k], want) <= TOL
            assert _err(ya[k], oracle.propagate(u[k], PITCH, 6e-6, LAM, 0.08, kind, of | oracle.ADJOINT)) <= TOL
            assert _err(yz[k], oracle.propagate(u[k], PITCH, 6e-6, LAM, 0.05 + 0.03 * k, kind, of)) <= TOL


@pytest.mark.parametrize("nx,ny", SHAPES)
def test_stacks_items_epilogues(cwo, nx, ny):
    import torch
    u = _fields(nx, ny, 4, nx)
    x = torch.from_numpy(u).cuda()
    zs = [0.04, 0.09, 0.15]
    for kind in (0, 1):
        plan = cwo.Plan(nx, ny, PITCH, PITCH, LAM, 0.1, kind)
        s = plan.propagate_stack(x[0], zs)
        inten = plan.propagate_epilogue(x, cwo.EPI_INTENSITY)
        plan.check()
        for k, z in enumerate(zs):
            assert _err(s[k], oracle.propagate(u[0], PITCH, PITCH, LAM, z, kind)) <= TOL
        want = np.abs(oracle.propagate(u[3], PITCH, PITCH, LAM, 0.1, kind)) ** 2
        assert _err(inten[3], want) <= 2 * TOL
    items = [dict(type=k % 2, z=0.03 + 0.02 * k, wavelength=LAM, dx=PITCH, dy=7e-6) for k in range(4)]
    y = plan.propagate_items(x, items)
    yo = plan.propagate_items(x, items, out=_off16(torch, x))
    plan.check()
    for k, it in enumerate(items):
        want = oracle.propagate(u[k], PITCH, 7e-6, LAM, it["z"], it["type"])
        assert _err(y[k], want) <= TOL and _err(yo[k], want) <= TOL
        assert torch.equal(plan.propagate_items(x[k:k + 1], items[k:k + 1])[0], y[k])
    own = cwo.Plan(nx, ny, PITCH, 7e-6, LAM, items[1]["z"], 1)
    assert torch.equal(own.propagate(x[1]), y[1])


@pytest.mark.parametrize("nx,ny", SHAPES)
def test_shifted_types(cwo, nx, ny):
    import torch
    u = _fields(nx, ny, 2, ny)
    x = torch.from_numpy(u).cuda()
    sh = (150e-6, -90e-6, 4e3, 1.2e5, -2e3, 1.1e5)
    for flags in (0, cwo.FLAG_PHASE_FP64):
        plan = cwo.Plan(nx, ny, PITCH, PITCH, LAM, 0.06, flags=flags, shift=cwo.Shift(*sh))
        y, ya = plan.propagate_batch(x), plan.propagate_batch(x, adjoint=True)
        plan.check()
        assert _err(y[1], oracle.propagate_shifted(u[1], PITCH, PITCH, LAM, 0.06, *sh)) <= TOL
        assert _err(ya[0], oracle.propagate_shifted(u[0], PITCH, PITCH, LAM, 0.06, *sh, flags=oracle.ADJOINT)) <= TOL
    prm = (6e-6, 4e-6, 0.0, 10e-6, 200e-6, -120e-6)
    plan = cwo.Plan(nx, ny, PITCH, PITCH, LAM, 0.3, shifted_fresnel=cwo.ShiftedFresnel(*prm))
    y = plan.propagate_batch(x)
    yo = plan.propagate_batch(x, out=_off16(torch, x))   # three passes
    ya = plan.propagate_batch(x, adjoint=True)
    plan.check()
    want = oracle.shifted_fresnel(u[1], PITCH, PITCH, prm[0], prm[1], LAM, 0.3, *prm[2:])
    assert _err(y[1], want) <= TOL and _err(yo[1], want) <= TOL
    lhs = torch.vdot(x[0].flatten().to(torch.complex128), y[1].flatten().to(torch.complex128))
    rhs = torch.vdot(ya[0].flatten().to(torch.complex128), x[1].flatten().to(torch.complex128))
    assert abs(complex(lhs - rhs)) <= 1e-5 * float(y[1].norm()) * float(x[0].norm())
