"""Refinement of the MP coefficients on a fixed support (differentiable
synthesis + SSIM).

The support -- leaves and atom indices of an encode -- is held fixed and the
coefficients are refined by gradient ascent on the mean SSIM (Section 3) of
the synthesised planes (Algorithm 3).  Forward and backward both run in the
library's kernels (`aqmp_refine_forward` / `aqmp_refine_backward`); this module only wraps them as a torch.autograd.Function.  The
loss uses the unclipped reconstruction (the clip of the reported metric has
no useful gradient where it saturates).
"""
from __future__ import annotations

import torch

from . import aqmp


class SynthesisSSIM(torch.autograd.Function):
    """mean over planes of SSIM(ref_p, synthesis_p(alpha)); alpha is the
    code's coefficient vector in canonical order (float32, CUDA)."""

    @staticmethod
    def forward(ctx, alpha, code, refs):
        # When alpha needs a gradient, the SSIM kernels return d SSIM / d y
        # in the same pass (the window statistics are computed once); the
        # backward only scales it and runs the synthesis adjoint.  All planes
        # go through one launch of each kernel.
        want = ctx.needs_input_grad[0]
        dev = alpha.device
        refs = list(refs)                        # walked several times
        at = [0]
        for _, ref in refs:
            at.append(at[-1] + ref.shape[0] * ref.shape[1])
        recon = torch.empty(at[-1], dtype=torch.float32, device=dev)
        grad = torch.empty_like(recon) if want else None
        y0, g0 = recon.data_ptr(), grad.data_ptr() if want else None
        planes = aqmp.aqmp_refine_planes([
            (plane, ref.shape[0], ref.shape[1], ref.data_ptr(), ref.stride(0), y0 + 4 * o, ref.shape[1],
             g0 + 4 * o if want else None, ref.shape[1]) for (plane, ref), o in zip(refs, at)])
        ssim = torch.empty(len(refs), dtype=torch.float64, device=dev)
        work = torch.empty(aqmp.aqmp_refine_workspace(planes), dtype=torch.uint8, device=dev) if want else None
        aqmp.aqmp_refine_forward(code, alpha, planes, ssim, work)
        # for the backward: the gradient images and where each plane's is (the
        # synthesis, the workspace and the references are not kept)
        ctx.code, ctx.images = code, grad
        ctx.sizes = [(plane, ref.shape[0], ref.shape[1]) for plane, ref in refs]
        ctx.n_alpha = alpha.shape[0]
        return ssim.mean()

    @staticmethod
    def backward(ctx, grad):
        grad_alpha = torch.zeros(ctx.n_alpha, dtype=torch.float32, device=grad.device)
        rows, at = [], ctx.images.data_ptr()
        for plane, h, w in ctx.sizes:
            rows.append((plane, h, w, None, 0, None, 0, at, w))
            at += 4 * h * w
        aqmp.aqmp_refine_backward(ctx.code, aqmp.aqmp_refine_planes(rows), grad_alpha)
        # the mean over planes and the upstream gradient, on the device
        return grad_alpha * (grad / len(ctx.sizes)).to(torch.float32), None, None


def synthesis_ssim(alpha, code, refs):
    return SynthesisSSIM.apply(alpha, code, refs)


def refine(code, refs, steps: int = 50, lr: float = 0.25):
    """`steps` Adam steps of SSIM ascent from the code's own coefficients.
    `refs` is a list of (plane index, reference image as CUDA float32).
    Returns (refined alpha, SSIM history with the starting value first)."""
    _, alpha0 = aqmp.aqmp_device_atoms(code)
    alpha = alpha0.clone().requires_grad_(True)
    opt = torch.optim.Adam([alpha], lr=lr)
    history = []
    for _ in range(steps):
        opt.zero_grad(set_to_none=True)
        s = synthesis_ssim(alpha, code, refs)
        (-s).backward()
        history.append(float(s.detach()))
        opt.step()
    with torch.no_grad():
        history.append(float(synthesis_ssim(alpha, code, refs)))
    return alpha.detach(), history
