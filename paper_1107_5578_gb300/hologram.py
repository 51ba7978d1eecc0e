"""Phase-only hologram optimisation through the differentiable propagation.

A phase phi [h][w] (1080 x 1920 by default) drives a unit-amplitude field exp(i phi), placed at
the centre of a square canvas of zeros (2048^2); the angular spectrum method (padded by the
library to 4096^2) propagates it by z, and the loss is the mean squared difference between the
intensity |U|^2 on the phi-sized window and a smooth target.  Adam updates phi; gradients come
from the hand-written adjoint kernel (autograd.propagate).

Usable as a module (HologramProblem, optimise) or as a script:
    python -m paper_1107_5578_gb300.hologram --steps 200
"""
from __future__ import annotations

import argparse
import json
import time

import numpy as np
import torch

from . import autograd, cwo, synth


_F32, _C64 = torch.float32, torch.complex64


class _Geometry:
    """The window of a problem on its canvas and the plan that propagates it, as they were at the call."""
    __slots__ = ("plan", "window", "canvas", "shapes")

    def __init__(self, p: "HologramProblem"):
        self.plan, self.canvas = p.plan, p.canvas
        h, w = p.h, p.w
        self.window = (h, w, p.ox, p.oy)
        self.shapes = ((h, w), (h, w), (p.canvas, p.canvas))   # of phase, gradient and field

    def forward(self, phi, target):
        """(u, |u|^2) of u = A exp(i phi), or, with a target, (u, residual, loss)"""
        phi = phi.contiguous()
        u = torch.empty(self.canvas, self.canvas, dtype=torch.complex64, device=phi.device)
        image = torch.empty(phi.shape, dtype=torch.float32, device=phi.device)
        if target is None:
            _call("cwo_hologram_forward", self.plan.handle, phi.data_ptr(), None, *self.window, u.data_ptr(), image.data_ptr(), None, None)
            return u, image
        loss = torch.empty((), dtype=torch.float32, device=phi.device)
        partial = torch.empty(cwo.HOLOGRAM_PARTIALS, dtype=torch.float64, device=phi.device)
        _call("cwo_hologram_forward", self.plan.handle, phi.data_ptr(), target.data_ptr(), *self.window, u.data_ptr(), image.data_ptr(),
              loss.data_ptr(), partial.data_ptr())
        return u, image, loss

    def backward(self, phi, u, g, gloss):
        """derivative by the phase, through the adjoint kernels"""
        # saved-tensor hooks may hand back another type than they were given
        if phi.dtype is not _F32 or g.dtype is not _F32 or u.dtype is not _C64:
            phi, u, g = phi.float(), u.to(_C64), g.float()
        if (phi.shape, g.shape, u.shape) != self.shapes:
            raise RuntimeError("a saved tensor came back with another shape")
        phi, u, g = phi.contiguous(), u.contiguous(), g.contiguous()
        work, out = torch.empty_like(u), torch.empty_like(phi)
        _call("cwo_hologram_backward", self.plan.handle, phi.data_ptr(), u.data_ptr(), g.data_ptr(),
              None if gloss is None else gloss.data_ptr(), *self.window, work.data_ptr(), out.data_ptr())
        return out

    # the same steps as tensor operators: for inputs the kernels do not take, and for gradients of
    # gradients
    def field(self, phi):
        h, w, ox, oy = self.window
        x = torch.zeros(self.canvas, self.canvas, dtype=torch.complex64, device=phi.device)
        x[oy:oy + h, ox:ox + w] = torch.polar(torch.ones_like(phi), phi)
        return x

    def intensity(self, phi):
        return self.field_intensity(self.field(phi))

    def field_intensity(self, x):
        h, w, ox, oy = self.window
        u = autograd.propagate(x, self.plan)
        uw = u[oy:oy + h, ox:ox + w]
        return uw.real ** 2 + uw.imag ** 2


def _call(name, *args):
    st = getattr(cwo.lib(), name)(*args, cwo._stream_handle(None))
    if st != cwo.OK:
        cwo.check(st, name)


class _Intensity(torch.autograd.Function):
    """phase [h][w] -> |A exp(i phase)|^2 on the window, through the fused kernels (cwo_holo.cu)."""

    @staticmethod
    def forward(ctx, phi, geo):
        u, image = geo.forward(phi, None)
        ctx.geo = geo
        ctx.save_for_backward(phi, u)
        return image

    @staticmethod
    def backward(ctx, gi):
        phi, u = ctx.saved_tensors
        if torch.is_grad_enabled():   # a graph of the gradient is wanted: the composed operators have one
            return torch.autograd.grad(ctx.geo.intensity(phi), phi, gi, create_graph=True)[0], None
        return ctx.geo.backward(phi, u, gi.resolve_neg(), None), None


class _Loss(torch.autograd.Function):
    """phase [h][w], target -> mean squared difference between the intensity and the target.  The
    residual is kept for the gradient, not the target, which the caller may change in the meantime."""

    @staticmethod
    def forward(ctx, phi, target, geo):
        u, residual, loss = geo.forward(phi, target)
        ctx.geo = geo
        ctx.save_for_backward(phi, u, residual)
        return loss

    @staticmethod
    def backward(ctx, gl):
        phi, u, residual = ctx.saved_tensors
        if torch.is_grad_enabled():
            inten = ctx.geo.intensity(phi)
            d = inten - (inten.detach() - residual)
            return torch.autograd.grad((d * d).mean(), phi, gl, create_graph=True)[0], None, None
        return ctx.geo.backward(phi, u, residual, gl.resolve_neg()), None, None


class HologramProblem:
    def __init__(self, h=1080, w=1920, canvas=2048, pitch=6.4e-6, wavelength=520e-9, z=0.15,
                 seed=1, device="cuda"):
        self.h, self.w, self.canvas = h, w, canvas
        self.oy, self.ox = (canvas - h) // 2, (canvas - w) // 2
        self.pitch, self.wavelength, self.z = pitch, wavelength, z
        self.device = torch.device(device)
        # every propagation of the optimisation has the same distance: the transfer function is kept (67
        # MB at 2048^2), except where the plan could then not propagate windows of rows
        self.plan = cwo.Plan(canvas, canvas, pitch, pitch, wavelength, z, cwo.ANGULAR, cwo.FLAG_CACHE_H if canvas < 4096 else 0)
        phi0, tgt = synth.hologram_problem(seed, h, w)
        self.phi0 = phi0
        # scale the target so that its energy matches the initial field's intensity on the window
        with torch.no_grad():
            i0 = self.intensity(torch.from_numpy(phi0).float().to(self.device))
        e0 = float(i0.sum())
        self.target_np = tgt * (e0 / float(tgt.sum()))
        self.target = torch.from_numpy(self.target_np).float().to(self.device)

    def field(self, phi: torch.Tensor) -> torch.Tensor:
        return _Geometry(self).field(phi)

    def _window(self, t) -> bool:
        """t is what the fused kernels take: a plain float32 CUDA tensor [h][w]"""
        return type(t) in (torch.Tensor, torch.nn.Parameter) and t.dtype == torch.float32 and t.is_cuda \
            and t.shape == (self.h, self.w) and not t.is_neg()

    # a step that a subclass, the instance or a patch of this class has replaced is called: the fused kernels do the
    # work of the ones below only
    def _fused(self, phi) -> bool:
        return getattr(self.field, "__func__", None) is _FIELD and self._window(phi) and self.plan.nx == self.plan.ny == self.canvas \
            and 0 <= self.oy <= self.canvas - self.h and 0 <= self.ox <= self.canvas - self.w

    def intensity(self, phi: torch.Tensor) -> torch.Tensor:
        geo = _Geometry(self)
        return _Intensity.apply(phi, geo) if self._fused(phi) else geo.field_intensity(self.field(phi))

    def loss(self, phi: torch.Tensor) -> torch.Tensor:
        geo, t = _Geometry(self), self.target
        if getattr(self.intensity, "__func__", None) is _INTENSITY and self._fused(phi) and self._window(t) and t.is_contiguous() and not t.requires_grad and t.device == phi.device:
            return _Loss.apply(phi, t, geo)
        d = self.intensity(phi) - t
        return (d * d).mean()


_FIELD, _INTENSITY = HologramProblem.field, HologramProblem.intensity


def optimise(problem: HologramProblem, steps=200, lr=0.05, log_every=0):
    phi = torch.from_numpy(problem.phi0).float().to(problem.device).requires_grad_(True)
    opt = torch.optim.Adam([phi], lr=lr)
    losses = []
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for s in range(steps):
        opt.zero_grad(set_to_none=True)
        L = problem.loss(phi)
        L.backward()
        opt.step()
        losses.append(L.detach())
        if log_every and (s % log_every == 0 or s == steps - 1):
            print(f"step {s:4d} loss {float(L.detach()):.6e}", flush=True)
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    return phi.detach(), [float(v) for v in losses], dt


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--lr", type=float, default=0.05)
    args = ap.parse_args()
    prob = HologramProblem()
    _, losses, dt = optimise(prob, args.steps, args.lr, log_every=20)
    print(json.dumps({"workload": "hologram_1920x1080_canvas2048_pad4096", "steps": args.steps,
                      "s_per_step": dt / args.steps, "loss_first": losses[0], "loss_last": losses[-1]}))


if __name__ == "__main__":
    main()
