"""torch.autograd.Function wrappers of the differentiable steps.

Forward and backward both run in the library's kernels (``libspp.so``);
these classes only allocate the output and gradient tensors and chain the
calls in the order of the chain rule:

    z --DensityToS--> s --Splat--> L^0..L^{L-1} --Reconstruct--> HDR, sRGB --L1Loss--> loss
                                          logits ----^

The discrete sampling decisions (counts, the sample list, the samples
themselves) are held fixed inside a step, as in the paper's relaxed
estimator (Sec. 4.3): gradients reach s through the 1/s normalisation and
the ramp weight, and reach the sampler logits z through the spatial softmax.
"""
from __future__ import annotations

import torch

from . import _binding as B


def _aligned(g):
    """An incoming gradient as the library takes it: contiguous, from a 16-byte
    boundary (a view into a larger tensor need not start at one); None stays None."""
    if g is None:
        return None
    g = g.contiguous()
    return g.clone() if g.data_ptr() % 16 else g


class Reconstruct(torch.autograd.Function):
    """Coarse-to-fine gather pyramid (Appendix A) with the tone map of Sec. 5.

    apply(L, tm, prev_warp, mask, *layers, *logits) -> (hdr, ldr)
    prev_warp: W_t L_{t-1} at full resolution (spp_warp_previous) or None.
    """

    @staticmethod
    def forward(ctx, L, tm, warped, mask, *tensors):
        layers, logits = list(tensors[:L]), list(tensors[L:2 * L])
        _, H, W = layers[0].shape
        hats = [None] + [torch.empty_like(x) for x in layers[1:]]
        hdr = torch.empty_like(layers[0])
        ldr = torch.empty_like(layers[0])
        B.check(B.spp_reconstruct_pyramid(layers, logits, warped,
                                          mask if warped is not None else None, W, H, tm, hats,
                                          hdr, ldr), "reconstruct")
        ctx.L, ctx.tm = L, tm
        # an output that the loss does not use needs no gradient of zeros
        ctx.set_materialize_grads(False)
        ctx.save_for_backward(warped if warped is not None else torch.empty(0, device=hdr.device),
                              mask if mask is not None else torch.empty(0, device=hdr.device,
                                                                        dtype=torch.uint8),
                              hdr, *layers, *logits, *hats[1:])
        ctx.has_warped = warped is not None
        ctx.has_mask = mask is not None
        return hdr, ldr

    @staticmethod
    def backward(ctx, g_hdr, g_ldr):
        L = ctx.L
        saved = ctx.saved_tensors
        warped = saved[0] if ctx.has_warped else None
        mask = saved[1] if ctx.has_mask else None
        hdr = saved[2]
        layers = list(saved[3:3 + L])
        logits = list(saved[3 + L:3 + 2 * L])
        hats = [None] + list(saved[3 + 2 * L:])
        _, H, W = hdr.shape
        new = lambda ts: [torch.empty_like(x) for x in ts]
        g_layers, g_logits, g_hats = new(layers), new(logits), [None] + new(hats[1:])
        g_warped = torch.empty_like(hdr) if warped is not None else None
        B.check(B.spp_reconstruct_pyramid_backward(
            layers, logits, hats, warped, mask, hdr, W, H, ctx.tm, _aligned(g_hdr),
            _aligned(g_ldr), torch.empty_like(hdr), g_layers, g_logits, g_hats, g_warped),
            "reconstruct backward")
        return (None, None, g_warped, None, *g_layers, *g_logits)


class WarpPrevious(torch.autograd.Function):
    """W_t L_{t-1} (App. A, Eq. app-recon-full)."""

    @staticmethod
    def forward(ctx, prev, mv):
        _, H, W = prev.shape
        out = torch.empty_like(prev)
        B.check(B.spp_warp_previous(prev, mv, W, H, out), "warp")
        ctx.save_for_backward(mv)
        return out

    @staticmethod
    def backward(ctx, g):
        (mv,) = ctx.saved_tensors
        _, H, W = g.shape
        g = _aligned(g)
        gp = torch.zeros_like(g)
        B.check(B.spp_warp_previous_backward(mv, W, H, g, gp), "warp backward")
        return gp, None


class L1Loss(torch.autograd.Function):
    """Mean |ldr - ref| (Eq. loss_spatial with the masking term m = 1)."""

    @staticmethod
    def forward(ctx, ldr, ref):
        loss = torch.empty(4, device=ldr.device)[:1]
        grad = torch.empty_like(ldr)
        B.check(B.spp_l1_loss(ldr, ref, ldr.numel(), loss, grad), "l1")
        ctx.save_for_backward(grad)
        return loss[0]

    @staticmethod
    def backward(ctx, g):
        (grad,) = ctx.saved_tensors
        return grad * g, None


class Splat(torch.autograd.Function):
    """The noisy pyramid as a function of the density s (Eq. stoch_rnoisy,
    Eq. app-pyramid), the samples and discrete choices of ``frame`` fixed.

    apply(frame, params, s) -> tuple of L layers (those computed by the last
    frame.splat() call)."""

    @staticmethod
    def forward(ctx, frame, params, s):
        ctx.frame, ctx.params, ctx.s_shape = frame, params, s.shape
        return tuple(x.clone() for x in frame.layers)

    @staticmethod
    def backward(ctx, *g_layers):
        fr, p = ctx.frame, ctx.params
        g0 = (g_layers[0].contiguous().clone() if g_layers[0] is not None
              else torch.zeros_like(fr.layers[0]))
        full = [g if g is not None else torch.zeros_like(x) for g, x in zip(g_layers, fr.layers)]
        full = [_aligned(x) for x in full]
        B.check(B.spp_pyramid_backward(full, fr.W, fr.H, fr.L, g0), "pyramid backward")
        gs = torch.empty_like(fr.s)
        B.check(B.spp_splat_backward(fr.offsets, fr.counts, fr.rgb, fr.s, fr.layers[0], g0,
                                     fr.capacity, fr.W, fr.H, p, gs), "splat backward")
        return None, None, gs.view(ctx.s_shape)


class DensityToS(torch.autograd.Function):
    """s = phi B + (1 - phi) B N softmax(z) (Sec. 3), given d = exp(z - max z).

    apply(d, s, budget, phi, z) -> s (the tensor the allocation wrote)."""

    @staticmethod
    def forward(ctx, d, s, budget, phi, z):
        ctx.save_for_backward(d)
        ctx.budget, ctx.phi = budget, phi
        return s.view_as(z).clone()

    @staticmethod
    def backward(ctx, g):
        (d,) = ctx.saved_tensors
        gz = torch.empty_like(d)
        ws = torch.empty(max(B.spp_density_backward_workspace_bytes(), 16), dtype=torch.uint8,
                         device=d.device)
        B.check(B.spp_density_backward(d, d.numel(), ctx.budget, ctx.phi, _aligned(g), gz, ws),
                "density backward")
        return None, None, None, None, gz.view_as(g)
