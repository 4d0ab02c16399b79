"""Weight gradient at the edges of its chunks: 64 pixels of a row, 32-channel
blocks of the input and of the gradient.

Against the FP64 oracle; the tolerance is the FP32 accumulation bound
(pixels/16 + 64) 2^-24 sum |x g| with a factor 4, as for the other shapes.
"""
import numpy as np
import pytest
import torch

import oracle.unet as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def spp():
    from conftest import build_spp_lib
    build_spp_lib()
    import paper_2602_08642_gb300 as spp
    torch.cuda.set_device(0)
    return spp


@pytest.mark.parametrize("B,H,W", [(1, 1, 1), (1, 4, 64), (2, 3, 63), (1, 5, 65), (3, 9, 130)])
@pytest.mark.parametrize("cin,cout", [(8, 8), (32, 32), (40, 24), (64, 72), (96, 32), (96, 96),
                                      (192, 128)])
def test_weight_gradient_tile_edges(spp, B, H, W, cin, cout):
    g = torch.Generator().manual_seed(1000 * cin + 10 * cout + W)
    x = torch.randn(B, H, W, cin, generator=g).to(torch.bfloat16)
    gy = torch.randn(B, H, W, cout, generator=g).to(torch.bfloat16)
    n = spp.binding.spp_conv3x3_backward_weights_workspace_bytes(B, W, H, cin, cout)
    ws = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")  # NaN where unwritten
    gw = torch.full((cout, cin, 3, 3), float("nan"), device="cuda")
    gb = torch.full((cout,), float("nan"), device="cuda")
    st = torch.zeros(4, dtype=torch.int32, device="cuda")[:1]
    spp.check(spp.binding.spp_conv3x3_backward_weights(x.cuda(), gy.cuda(), B, W, H, cin, cout, gw,
                                                       gb, ws, st))
    assert spp.binding.spp_get_status(st) == 0
    nchw = lambda t: t.float().numpy().astype(np.float64).transpose(0, 3, 1, 2)
    xb, gyb = nchw(x), nchw(gy)
    w0 = np.zeros((cout, cin, 3, 3))
    ref_w = sum(U.conv3x3_backward(xb[b], w0, gyb[b])[1] for b in range(B))
    abs_w = sum(U.conv3x3_backward(np.abs(xb[b]), w0, np.abs(gyb[b]))[1] for b in range(B))
    tol = 4 * (B * H * W / 16 + 64) * 2.0 ** -24
    assert np.all(np.abs(gw.cpu().numpy() - ref_w) <= tol * abs_w)
    assert np.all(np.abs(gb.cpu().numpy() - gyb.sum(axis=(0, 2, 3)))
                  <= tol * np.abs(gyb).sum(axis=(0, 2, 3)))


@pytest.mark.parametrize("W", [1, 2, 7, 8, 16, 20, 24, 44, 48, 63, 64, 65, 70, 80, 130])
@pytest.mark.parametrize("cin,cout", [(32, 32), (40, 72), (192, 128)])
def test_infinities_stay_with_the_taps_that_read_them(spp, W, cin, cout):
    """The first and last input pixels of a row have no output pixel to their right
    (tap dx = 2) and to their left (dx = 0): an infinity or NaN there leaves those
    taps as they are with a 0 in its place, the same bits."""
    B, H = 2, 3
    g = torch.Generator().manual_seed(100 * cin + W)
    x = torch.randn(B, H, W, cin, generator=g).to(torch.bfloat16)
    gy = torch.randn(B, H, W, cout, generator=g).to(torch.bfloat16).cuda()
    bad = x.clone()
    for c, v in ((1, float("inf")), (cin // 2, float("nan")), (cin - 1, -float("inf"))):
        x[:, :, -1, c] = 0
        bad[:, :, -1, c] = v
        if W > 1:
            x[:, 1, 0, c - 1] = 0
            bad[:, 1, 0, c - 1] = v
    got = []
    for t in (x, bad):
        n = spp.binding.spp_conv3x3_backward_weights_workspace_bytes(B, W, H, cin, cout)
        ws = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")
        gw = torch.full((cout, cin, 3, 3), float("nan"), device="cuda")
        gb = torch.full((cout,), float("nan"), device="cuda")
        spp.check(spp.binding.spp_conv3x3_backward_weights(t.cuda(), gy, B, W, H, cin, cout, gw, gb,
                                                           ws, None))
        got.append((gw.cpu().numpy(), gb.cpu().numpy()))
    (gw, gb), (bw, bb) = got
    last = [1, cin // 2, cin - 1]
    first = [c - 1 for c in last] if W > 1 else []
    clean = [c for c in range(cin) if c not in last + first]
    assert np.all(np.isfinite(gw)) and np.array_equal(gb, bb)
    assert np.array_equal(gw[:, clean], bw[:, clean])
    assert np.array_equal(gw[:, last][..., 0], bw[:, last][..., 0])
    assert np.array_equal(gw[:, first][..., 2], bw[:, first][..., 2])
    assert not np.isfinite(bw[:, last][:, :, 1, 1]).any()
