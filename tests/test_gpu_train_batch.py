"""A training step with one launch per step of the renderer for the whole
batch against the same step sample by sample.

Both run the same kernels on the same values in the same order per image, so
parameters, gradients and images are the same bits; the loss sums blocks with
atomics and is held to FP32 rounding of its few hundred terms (1e-5).
"""
import numpy as np
import pytest
import torch

import spp_inputs as inp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Lm():
    from conftest import build_spp_lib
    build_spp_lib()
    from paper_2602_08642_gb300 import learned
    torch.cuda.set_device(0)
    return learned


@pytest.mark.parametrize("batch,size,kw", [
    (1, 20, {}), (3, 64, {}), (2, 24, dict(objective="combined", random_tmo=True)),
    (17, 16, {}),                                   # more images than one launch takes
    (2, 72, dict(estimator="straight_through")), (2, 40, dict(estimator="gumbel")),
    (2, 32, dict(estimator="dasr")), (3, 64, dict(dither=True))])
def test_batched_step_matches_sample_by_sample(Lm, batch, size, kw):
    kw = dict(kw)
    mask = None
    if kw.pop("dither", False):
        mask = torch.from_numpy(Lm.B.spp_blue_noise_mask(16, 3).view(np.int16)).cuda()
    theta = torch.from_numpy(inp.unet_params(Lm.layer_table(), seed=5, head_scale=0.3,
                                             head_bias=inp.fixed_head_bias()))
    samples = [Lm.FrameData(inp.training_pair(size, seed=50 + k), seed=k) for k in range(batch)]
    got = []
    for batched in (True, False):
        tr = Lm.Trainer(theta, batch, size, 0.4, lr=1e-3, dither_mask=mask, **kw)
        assert tr.rnd.batched
        tr.rnd.batched = batched
        losses = [tr.step(samples, 900 + 40 * k) for k in range(2)]
        assert all(fr.check_status() == 0 for fr in tr.rnd.frames)
        got.append((losses, [tr.net.theta, tr.net.grad, *tr.rnd.ldr, *tr.rnd.hdr_prev,
                             *[fr.counts for fr in tr.rnd.frames],
                             *[fr.s for fr in tr.rnd.frames]]))
    assert np.allclose(got[0][0], got[1][0], rtol=1e-5)
    for a, b in zip(got[0][1], got[1][1]):
        assert torch.equal(a, b)


def test_part_of_a_batch_and_unaligned_sizes(Lm):
    """Fewer samples than the batch take the step sample by sample; a size
    whose coarsest images do not start on 16-byte boundaries is refused as
    before for more than one sample, and taken for one."""
    theta = torch.from_numpy(inp.unet_params(Lm.layer_table(), seed=5, head_scale=0.3,
                                             head_bias=inp.fixed_head_bias()))
    samples = [Lm.FrameData(inp.training_pair(64, seed=50), seed=0)]
    assert np.isfinite(Lm.Trainer(theta, 2, 64, 0.4).step(samples, 1))
    odd = [Lm.FrameData(inp.training_pair(20, seed=50 + k), seed=k) for k in range(2)]
    assert np.isfinite(Lm.Trainer(theta, 1, 20, 0.4).step(odd[:1], 1))
    with pytest.raises(Lm.B.SppError):
        Lm.Trainer(theta, 2, 20, 0.4).step(odd, 1)


def test_expired_waits_reach_the_status_of_their_images(Lm):
    """A reconstruction tile whose copies never arrive: the status of every image
    with a tile that its block then leaves out says so, and no other's."""
    B, n, W, H = Lm.B, 3, 128, 128  # 64 tiles of 64 x 4 pixels per image
    tiles = (W // 64) * (H // 4)
    G = min(torch.cuda.get_device_properties(0).multi_processor_count, n * tiles)
    g = torch.Generator(device="cuda").manual_seed(3)
    noisy, logits = (torch.randn(n, c, H, W, generator=g, device="cuda") for c in (3, 25))
    out, st = torch.empty_like(noisy), torch.zeros(n, 4, dtype=torch.int32, device="cuda")
    for stalled in (30, tiles + 1, n * tiles - 1):
        st.zero_()
        assert B.spp_test_stall_reconstruction(stalled) == 0
        B.check(B.spp_reconstruct_level_batch(n, noisy, logits, 25, None, None, None, W, H, None,
                                              out, None, st))
        left_out = {t // tiles for t in range(stalled, n * tiles, G)}
        assert [c != 0 for c in st[:, 0].tolist()] == [b in left_out for b in range(n)]
        assert not st[:, 1:].any()

    # the previous frames of a training step report to their frames
    rnd = Lm.Renderer(2, 64, 64, 0.25)
    heads = [torch.zeros(2, c, 64 >> l, 64 >> l, device="cuda") for l, c in enumerate((55, 29, 25))]
    args = (torch.ones(2, 64, 64, device="cuda"), heads, [torch.ones(3, 64, 64, device="cuda")] * 2,
            5, 0)
    assert B.spp_test_stall_reconstruction(5) == 0  # level 2: tiles 4 to 7 are image 1's
    rnd.previous_frame_all(*args)
    assert rnd.frames[0].check_status() == 0
    with pytest.raises(B.SppError) as e:
        rnd.frames[1].check_status()
    assert e.value.code == B.SPP_ERR_TIMEOUT
    rnd.frames[1].clear_status()
    rnd.previous_frame_all(*args)
    assert all(fr.check_status() == 0 for fr in rnd.frames)


@pytest.mark.parametrize("objective", ["l1", "combined"])
def test_part_of_a_batch_is_that_part_only(Lm, objective):
    """A step of 2 samples on a trainer of 3, after a step of 3, against the same
    step on a trainer of 2 in the same state: the third image's gradients and loss
    of the step before take no part.  The two cut the weight gradients' sums
    differently, which shows in the 5th digit: 1e-3 of the gradient's norm; an
    image of the step before is of the norm's own size."""
    theta = torch.from_numpy(inp.unet_params(Lm.layer_table(), seed=5, head_scale=0.3,
                                             head_bias=inp.fixed_head_bias()))
    samples = [Lm.FrameData(inp.training_pair(64, seed=50 + k), seed=k) for k in range(3)]
    a = Lm.Trainer(theta, 3, 64, 0.4, objective=objective)
    a.step(samples, 900)
    b = Lm.Trainer(theta, 2, 64, 0.4, objective=objective)
    for name in ("theta", "m", "v"):
        getattr(b.net, name).copy_(getattr(a.net, name))
    b.net.step_count, b.step_index = a.net.step_count, a.step_index
    b.net.pack()
    la, lb = a.step(samples[:2], 940), b.step(samples[:2], 940)
    assert abs(la - lb) <= 1e-5 * lb
    assert torch.linalg.norm(a.net.grad - b.net.grad) <= 1e-3 * torch.linalg.norm(b.net.grad)
