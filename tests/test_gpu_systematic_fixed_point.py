"""The systematic sample map's integer path against its FP64 path.

SPP_FLAG_EXACT_FP64 makes every pixel run the FP64 sequence; without it
integers decide the pixels that are clear of a rounding boundary.  Counts,
offsets, sample list, s and holdout weights are the same bits, over the forms
that the entry accepts: budgets, uniform shares, slopes of the ramp, the hard
rule, densities over many binades, zeros and subnormals, ragged sizes.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def spp():
    from conftest import build_spp_lib
    build_spp_lib()
    import paper_2602_08642_gb300 as spp
    torch.cuda.set_device(0)
    return spp


def _density(kind, W, H):
    r = np.random.default_rng(W * 7 + H)
    if kind == "lognormal":
        d = np.exp(r.standard_normal((H, W)))
    elif kind == "wide":  # 150 binades, with zeros and subnormals
        d = np.exp2(r.uniform(-140, 10, (H, W))) * (r.random((H, W)) > 0.05)
        d.flat[0] = 1.0
    else:  # few values, so that many s_i sit on or next to rounding boundaries
        d = r.integers(0, 5, (H, W)).astype(np.float64)
        d.flat[0] = 1.0
    return torch.from_numpy(d.astype(np.float32)).cuda()


@pytest.mark.parametrize("W,H", [(1, 1), (7, 3), (130, 61), (1000, 333)])
@pytest.mark.parametrize("kind", ["lognormal", "wide", "steps"])
@pytest.mark.parametrize("budget,phi,lam,hard", [
    (0.25, 0.125, 10.0, False), (0.11, 0.0, 1.0, False), (4.0, 0.5, 1e6, False),
    (300.0, 1.0, 3.0, False), (0.5, 0.125, 10.0, True)])
def test_integer_path_matches_fp64_path(spp, W, H, kind, budget, phi, lam, hard):
    d = _density(kind, W, H)
    got = []
    for exact in (False, True):
        fr = spp.Frame(W, H, 1, max_budget=budget + 1.0, capacity=int((budget + 2) * W * H) + 64)
        fr.sample_pixel.fill_(-1)
        fr.alloc_systematic(d, spp.binding.make_params(budget, uniform_fraction=phi, lam=lam,
                                                       seed=11, frame=2, hard=hard,
                                                       exact_fp64=exact))
        assert fr.check_status() == 0
        got.append([t.cpu().numpy().copy() for t in (fr.counts, fr.offsets, fr.sample_pixel, fr.s,
                                                     fr.holdout_w, fr.total)])
    for a, b in zip(*got):
        assert np.array_equal(a.view(np.uint32 if a.dtype == np.float32 else a.dtype),
                              b.view(np.uint32 if b.dtype == np.float32 else b.dtype))


@pytest.mark.parametrize("N,budget,phi,base,spikes", [
    (1000, 600.0, 0.5, 297.78, [4020.0]),
    (1000, 600.0, 0.5, 297.0, [3000.0, 3790.0, 3800.0, 3900.0, 4000.0, 4050.0]),
    (64, 1500.0, 0.6, 600.0, [3900.0, 4000.0, 4090.0]),
    (5000, 900.0, 0.9, 90.0, [3100.0, 3300.0, 4000.0, 4095.0]),
    (333, 1023.0, 0.9, 66.6, [4000.0, 4060.0, 4095.0])])
def test_pixels_around_4096_samples(spp, N, budget, phi, base, spikes):
    """A uniform share on top of a product just under 4096 passes 2^64 in units of
    2^-52: those pixels, and their neighbours below and above, are the FP64
    sequence's, and the frame keeps its exact total."""
    d = torch.full((1, N), base, device="cuda")
    for k, v in enumerate(spikes):
        d[0, (k + 1) * N // (len(spikes) + 1)] = v
    got = []
    for exact in (False, True):
        fr = spp.Frame(N, 1, 1, max_budget=budget + 1.0, capacity=int((budget + 2) * N) + 64)
        fr.sample_pixel.fill_(-1)
        fr.alloc_systematic(d, spp.binding.make_params(budget, uniform_fraction=phi, seed=11,
                                                       frame=2, exact_fp64=exact))
        assert fr.check_status() == 0
        got.append([t.cpu().numpy().copy() for t in (fr.counts, fr.offsets, fr.sample_pixel, fr.s,
                                                     fr.holdout_w, fr.total)])
    assert got[1][3].max() > 3000 and abs(int(got[0][5][0]) - round(budget * N)) <= 1
    for a, b in zip(*got):
        assert np.array_equal(a.view(np.uint32 if a.dtype == np.float32 else a.dtype),
                              b.view(np.uint32 if b.dtype == np.float32 else b.dtype))
