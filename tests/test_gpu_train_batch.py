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
