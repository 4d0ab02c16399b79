"""Per-frame driver of the plain method over the C ABI.

Holds the device buffers of one W x H frame (PyTorch allocates them; the
library allocates nothing) and runs the steps of the hot path in order:
sample-count map and sample list, renderer stand-in, splat + pyramid,
coarse-to-fine reconstruction with the temporal term and the tone map.
Every step is a call into ``libspp.so``; this module only sizes buffers and
passes pointers.
"""
from __future__ import annotations

import math

import torch

from . import _binding as B


def logit_channels(level: int, L: int, temporal: bool) -> int:
    if level == L - 1:
        return 25
    if level == 0 and temporal:
        return 54
    return 29


def default_capacity(W: int, H: int, max_budget: float) -> int:
    """Sample slots for a frame: the budget plus a wide statistical margin
    (T is a sum of independent Bernoulli draws around B N)."""
    N = W * H
    return int(max_budget * N + 8.0 * math.sqrt(max(N, 1)) + 4096)


class Frame:
    """Device buffers for W x H frames with an L-level pyramid."""

    def __init__(self, W: int, H: int, L: int, *, max_budget: float = 0.5,
                 capacity: int | None = None, device: str | torch.device = "cuda",
                 storage: dict | None = None):
        """storage: buffers to use instead of new ones, by attribute name (the
        images of a FrameBatch share theirs)."""
        self.W, self.H, self.L = W, H, L
        self.N = N = W * H
        self.device = torch.device(device)
        dev = self.device
        self.capacity = capacity if capacity is not None else default_capacity(W, H, max_budget)
        i32, f32 = torch.int32, torch.float32
        st = storage or {}
        new = lambda name, shape, dtype: (st[name] if name in st else
                                          torch.empty(shape, dtype=dtype, device=dev))
        self.counts = new("counts", N, i32)
        self.offsets = new("offsets", N + 1, i32)
        self.sample_pixel = new("sample_pixel", max(self.capacity, 1), i32)
        self.s = new("s", N, f32)
        self.holdout_w = new("holdout_w", N, f32)
        self.total = st["total"] if "total" in st else torch.zeros(2, dtype=torch.int64,
                                                                   device=dev)[:1]
        self.status = st["status"] if "status" in st else torch.zeros(4, dtype=i32, device=dev)[:1]
        self.alloc_ws = new("alloc_ws", max(B.spp_alloc_workspace_bytes(W, H), 16), torch.uint8)
        self.rgb = new("rgb", (max(self.capacity, 1), 4), f32)
        self.layers = st["layers"] if "layers" in st else [
            torch.empty((3, H >> l, W >> l), dtype=f32, device=dev) for l in range(L)]
        self.recon_ws = torch.empty(max(B.spp_reconstruct_workspace_bytes(W, H, L), 16),
                                    dtype=torch.uint8, device=dev)
        self.hdr = [torch.zeros((3, H, W), dtype=f32, device=dev) for _ in range(2)]
        self.ldr = torch.empty((3, H, W), dtype=f32, device=dev)
        self.parity = 0  # which hdr buffer receives the next output

    # ----------------------------------------------------------------- steps
    def alloc(self, d: torch.Tensor, params: B.spp_params, stream=None):
        B.check(B.spp_alloc_sample_map(d, self.W, self.H, params, self.counts, self.offsets,
                                       self.sample_pixel, self.capacity, self.s, self.holdout_w,
                                       self.total, self.status, self.alloc_ws, stream),
                "spp_alloc_sample_map")

    def alloc_dithered(self, d: torch.Tensor, params: B.spp_params, mask: torch.Tensor,
                       stream=None):
        """alloc with the uniforms from a blue-noise rank mask (device int16
        view of spp_blue_noise_mask's uint16 [T][T])."""
        B.check(B.spp_alloc_sample_map_dithered(d, self.W, self.H, params, mask, self.counts,
                                                self.offsets, self.sample_pixel, self.capacity,
                                                self.s, self.holdout_w, self.total, self.status,
                                                self.alloc_ws, stream),
                "spp_alloc_sample_map_dithered")

    def alloc_systematic(self, d: torch.Tensor, params: B.spp_params, stream=None):
        """alloc with systematic (exact-integer-total) rounding."""
        B.check(B.spp_alloc_sample_map_systematic(d, self.W, self.H, params, self.counts,
                                                  self.offsets, self.sample_pixel, self.capacity,
                                                  self.s, self.holdout_w, self.total,
                                                  self.status, self.alloc_ws, stream),
                "spp_alloc_sample_map_systematic")

    def render(self, clean: torch.Tensor, seed: int, frame: int, stream=None):
        B.check(B.spp_render_synthetic(clean, self.offsets, self.sample_pixel, self.total,
                                       self.capacity, self.W, self.H, seed, frame, self.rgb,
                                       stream), "spp_render_synthetic")

    def splat(self, stream=None):
        B.check(B.spp_splat_samples(self.offsets, self.rgb, self.s, self.holdout_w,
                                    self.capacity, self.W, self.H, self.L, self.layers, stream),
                "spp_splat_samples")

    def reconstruct(self, logits, prev=None, mv=None, mask=None, tm=None, stream=None):
        out = self.hdr[self.parity]
        C0 = logits[0].shape[0]
        B.check(B.spp_reconstruct_frame(self.layers, logits, C0, prev, mv, mask, self.W, self.H,
                                        self.L, tm if tm is not None else B.make_tonemap(), out,
                                        self.ldr, self.recon_ws, self.status, stream),
                "spp_reconstruct_frame")
        self.parity ^= 1
        return out

    def run(self, d, clean, logits, params: B.spp_params, *, render_seed: int = 0xC0FFEE,
            prev=None, mv=None, mask=None, tm=None, stream=None):
        """One frame of the plain method; returns the HDR output tensor."""
        self.alloc(d, params, stream)
        self.render(clean, render_seed, params.frame, stream)
        self.splat(stream)
        return self.reconstruct(logits, prev=prev, mv=mv, mask=mask, tm=tm, stream=stream)

    def check_status(self, stream=None) -> int:
        code = B.spp_get_status(self.status, stream)
        B.check(code, "device status")
        return code

    def clear_status(self, stream=None):
        B.check(B.spp_clear_status(self.status, stream), "spp_clear_status")

    def sample_count(self) -> int:
        return int(self.total.item())


class FrameBatch:
    """Device buffers of a batch of n frames of one size, held image after
    image as the batched entry points take them, and ``frames``, the n Frames
    whose buffers are parts of them.  Every image has to start on a 16-byte
    boundary on every level (``fits``)."""

    @staticmethod
    def fits(W: int, H: int, L: int) -> bool:
        return all((W >> l) * (H >> l) % 4 == 0 for l in range(L))

    def __init__(self, n: int, W: int, H: int, L: int, *, max_budget: float = 0.5,
                 device: str | torch.device = "cuda"):
        N = W * H
        # whole 16-byte pieces, for the images' sample lists too
        self.capacity = cap = -(-default_capacity(W, H, max_budget) // 4) * 4
        i32, f32 = torch.int32, torch.float32
        e = lambda *shape, dtype=f32: torch.empty(shape, dtype=dtype, device=device)
        self.counts = e(n, N, dtype=i32)
        self.offsets = e(n, N + B.SPP_BATCH_OFFSETS_PAD, dtype=i32)
        self.sample_pixel = e(n, cap, dtype=i32)
        self.s, self.holdout_w = e(n, N), e(n, N)
        self.total = torch.zeros(n, 2, dtype=torch.int64, device=device)
        self.status = torch.zeros(n, 4, dtype=i32, device=device)
        self.alloc_ws = e(B.spp_alloc_batch_workspace_bytes(n, W, H), dtype=torch.uint8)
        self.rgb = e(n, cap, 4)
        self.layers = [e(n, 3, H >> l, W >> l) for l in range(L)]
        ws = self.alloc_ws.view(n, -1)
        self.frames = [Frame(W, H, L, capacity=cap, device=device, storage=dict(
            counts=self.counts[b], offsets=self.offsets[b, :N + 1],
            sample_pixel=self.sample_pixel[b], s=self.s[b], holdout_w=self.holdout_w[b],
            total=self.total[b, :1], status=self.status[b, :1], alloc_ws=ws[b], rgb=self.rgb[b],
            layers=[x[b] for x in self.layers])) for b in range(n)]
