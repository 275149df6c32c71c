"""torch.autograd.Function over the batched fill and its hand-written adjoint.

    out = guidefill_fill(rgba, labels, mag, phi, mu, eps=3.0, c=0.05)
    loss = 0.5 * ((out - gt) ** 2).sum(); loss.backward()

rgba [B,H,W,4] float32, labels [B,H,W] uint8, guidance as magnitude mag [B,H,W]
and angle phi [B,H,W] (g = mag (cos phi, sin phi)), mu a 0-d tensor.
Gradients flow to rgba (the known colours), phi and mu; the shell schedule,
the stall steps and each ghost sample's tap set are held fixed (piecewise
constant).  Both passes run in libguidefill.so; the forward keeps only the shell
map, the stall bitmap, the guide field and its output for the backward.
"""
from __future__ import annotations

import torch

from . import context


_ONE_FIELD = 2 ** 31 - 64  # pixels that one guide field can have


class GuidefillFunction(torch.autograd.Function):
    @staticmethod
    def forward(ctx, rgba, labels, mag, phi, mu, eps, c):
        g = context(rgba.device.index)
        B = rgba.shape[0]
        muf = float(mu)
        if all(torch.is_tensor(t) and t.shape == rgba.shape[:3] for t in (labels, mag, phi)) and \
                0 < labels.numel() <= _ONE_FIELD:
            # one field B times as high: the conversion is per pixel
            H, W = labels.shape[1:]
            field = g.guide_from_angle(labels.reshape(B * H, W), mag.reshape(B * H, W), phi.reshape(B * H, W))
            guides = list(field.view(B, H, W, 2).unbind())
            labels = labels.unbind()
        else:  # lists of frames, batches longer than rgba's
            guides = [g.guide_from_angle(labels[i], mag[i], phi[i]) for i in range(B)]
            labels = [labels[i] for i in range(B)]
        # the frames' results are kept for the backward pass; the caller gets a copy to do
        # with as it likes (on the context's device: colours on the CPU are copied there)
        kept = torch.empty(tuple(rgba.shape[:3]) + (4,), dtype=torch.float32, device=torch.device("cuda", g.device))
        res = g.fill_batched(list(rgba.unbind()), labels, guides, eps=eps, mu=muf, c=c,
                             out=list(kept.unbind()), stall=True)
        out = kept.clone()
        ctx.res = res
        ctx.guides = guides
        ctx.eps, ctx.mu, ctx.c = eps, muf, c
        ctx.phi_tensor = torch.is_tensor(phi)  # a list of frames has no gradient
        ctx.mu_device = mu.device if torch.is_tensor(mu) else None
        return out

    @staticmethod
    def backward(ctx, grad_out):
        g = context(grad_out.device.index)
        B = grad_out.shape[0]
        grad_out = grad_out.contiguous()
        H, W = ctx.res[0].shell.shape
        dev = torch.device("cuda", g.device)
        grad_rgba = torch.empty((B, H, W, 4), dtype=torch.float32, device=dev)
        grad_phi = torch.empty((B, H, W), dtype=torch.float32, device=dev)
        _, _, gmu = g._backward(ctx.res, ctx.guides, list(grad_out.unbind()), eps=ctx.eps, mu=ctx.mu, c=ctx.c,
                                out=(grad_rgba.unbind(), grad_phi.unbind()))
        grad_mu = gmu.sum()
        if ctx.mu_device is not None:
            grad_mu = grad_mu.to(ctx.mu_device)
        return grad_rgba, None, None, grad_phi if ctx.phi_tensor else None, grad_mu, None, None


def guidefill_fill(rgba, labels, mag, phi, mu, eps=3.0, c=0.05):
    if not torch.is_tensor(mu):
        mu = torch.tensor(float(mu))
    return GuidefillFunction.apply(rgba, labels, mag, phi, mu, eps, c)
