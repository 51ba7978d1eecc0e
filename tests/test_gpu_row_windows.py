"""Propagations of row windows (cwo_propagate_rows): rows outside the input window are never read, rows outside
the output window never written, and the rest is what the whole field gives."""
import numpy as np
import pytest

from paper_1107_5578_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(16, 16), (64, 128), (256, 64), (512, 512), (2048, 1024), (4096, 64), (64, 4096)])
@pytest.mark.parametrize("cached", [False, True])
def test_windows(gpu, nx, ny, cached):
    import torch
    from paper_1107_5578_gb300 import cwo
    plan = cwo.Plan(nx, ny, 8e-6, 6e-6, 532e-9, 0.03, cwo.ANGULAR, cwo.FLAG_CACHE_H if cached else 0)
    g = plan.rows_group
    if cached and ny == 4096:
        assert g == 0
        with pytest.raises(cwo.CwoError):
            plan.propagate_rows(torch.zeros(ny, nx, dtype=torch.complex64, device="cuda"), (0, 8), (0, 8))
        return
    u = torch.from_numpy(synth.random_field(nx, seed=nx + ny, ny=ny).astype(np.complex64)).cuda()
    for ilo, ihi, olo, ohi in ((0, ny, 0, ny), (0, 1, ny - 1, ny), (ny // 3, ny // 2 + 1, ny // 4, ny // 4 + 3), (5, ny - 3, 9, ny)):
        x = torch.zeros_like(u)
        x[ilo:ihi] = u[ilo:ihi]
        for adjoint in (False, True):
            want = plan.adjoint(x) if adjoint else plan.propagate(x)
            xin = x.clone()
            lo, hi = ilo // g * g, -(-ihi // g) * g
            xin[:lo], xin[hi:] = float("nan"), float("nan")          # not read
            out = torch.full_like(x, 7.0)
            plan.propagate_rows(xin, (ilo, ihi), (olo, ohi), out=out, adjoint=adjoint)
            plan.check()
            lo, hi = olo // g * g, -(-ohi // g) * g
            # the same kernels on the same values; a transfer function evaluated in another instance of
            # the column kernel may round its phase once differently
            assert float((out[lo:hi] - want[lo:hi]).norm()) <= 1e-6 * float(want.norm())
            assert bool((out[:lo] == 7.0).all()) and bool((out[hi:] == 7.0).all())
    for bad in ((-1, 4, 0, 4), (0, ny + 1, 0, 4), (4, 4, 0, 4), (0, 4, 8, 8)):
        with pytest.raises(cwo.CwoError):
            plan.propagate_rows(u, bad[:2], bad[2:])
