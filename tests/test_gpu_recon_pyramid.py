"""The whole-pyramid calls against the same levels called one by one: equal
values, whatever the gradient buffers held before."""
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


@pytest.mark.parametrize("W,H,L,temporal", [(2, 2, 2, True), (36, 12, 2, True), (68, 20, 3, True),
                                            (30, 6, 2, False), (128, 32, 4, False)])
@pytest.mark.parametrize("use_hdr,use_ldr", [(True, True), (False, True), (True, False),
                                             (False, False)])
def test_pyramid_calls_equal_level_calls(spp, W, H, L, temporal, use_hdr, use_ldr):
    B = spp.binding
    g = torch.Generator(device="cuda").manual_seed(W * 100 + H)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    layers = [rnd(3, H >> l, W >> l).exp() for l in range(L)]
    # one plane more than needed at level 0: its gradient is 0
    logits = [rnd((55 if temporal else 30) if l == 0 else 25 if l == L - 1 else 29, H >> l, W >> l)
              for l in range(L)]
    warped = rnd(3, H, W).exp() if temporal else None
    mask = (rnd(H, W) > 1).to(torch.uint8) if temporal else None
    tm = B.make_tonemap()
    junk = lambda ts: [torch.full_like(t, float("nan")) for t in ts]

    hats = [None] + junk(layers[1:])
    hdr, ldr = junk([layers[0]] * 2)
    B.check(B.spp_reconstruct_pyramid(layers, logits, warped, mask, W, H, tm, hats, hdr, ldr))
    hats1 = [None] + junk(layers[1:])
    hdr1, ldr1 = junk([layers[0]] * 2)
    for l in range(L - 1, -1, -1):
        B.check(B.spp_reconstruct_level(
            layers[l], logits[l], logits[l].shape[0], hats1[l + 1] if l + 1 < L else None,
            warped if l == 0 else None, mask if l == 0 else None, W >> l, H >> l,
            tm if l == 0 else None, hdr1 if l == 0 else hats1[l], ldr1 if l == 0 else None))
    for a, b in zip([hdr, ldr] + hats[1:], [hdr1, ldr1] + hats1[1:]):
        assert torch.equal(a, b)

    g_hdr, g_ldr = rnd(3, H, W), rnd(3, H, W)
    gl, gz, gh = junk(layers), junk(logits), [None] + junk(hats[1:])
    gw = junk([hdr])[0] if temporal else None
    B.check(B.spp_reconstruct_pyramid_backward(
        layers, logits, hats, warped, mask, hdr, W, H, tm, g_hdr if use_hdr else None,
        g_ldr if use_ldr else None, junk([hdr])[0], gl, gz, gh, gw))
    out = g_hdr.clone() if use_hdr else torch.zeros_like(hdr)
    if use_ldr:
        B.check(B.spp_tonemap_backward(hdr, W, H, tm, g_ldr, out))
    gw1 = torch.zeros_like(hdr) if temporal else None
    for l in range(L):
        gl1, gz1 = torch.zeros_like(layers[l]), junk([logits[l]])[0]
        gc = torch.zeros_like(hats[l + 1]) if l + 1 < L else None
        B.check(B.spp_reconstruct_level_backward(
            layers[l], logits[l], logits[l].shape[0], hats[l + 1] if l + 1 < L else None,
            warped if l == 0 else None, mask if l == 0 else None, W >> l, H >> l, out, gz1, gl1, gc,
            gw1 if l == 0 else None))
        assert torch.equal(gl[l], gl1) and torch.equal(gz[l], gz1)
        if gc is not None:
            assert torch.equal(gh[l + 1], gc)
            out = gc
    if temporal:
        assert torch.equal(gw, gw1)


def test_gradient_views_of_any_alignment(spp):
    """The gradient of the HDR output may be a view that starts between 16-byte
    boundaries, or an expanded one."""
    from paper_2602_08642_gb300 import autograd
    W, H, L = 36, 12, 2
    g = torch.Generator(device="cuda").manual_seed(5)
    leaf = lambda *s: torch.randn(*s, generator=g, device="cuda").requires_grad_(True)
    layers = [leaf(3, H >> l, W >> l) for l in range(L)]
    logits = [leaf(29, H, W), leaf(25, H // 2, W // 2)]
    hdr, _ = autograd.Reconstruct.apply(L, spp.binding.make_tonemap(), None, None, *layers, *logits)
    inputs = layers + logits
    grads = lambda go: torch.autograd.grad(hdr, inputs, go, retain_graph=True)
    buf = torch.randn(3 * H * W + 1, generator=g, device="cuda")
    view = buf[1:].view(3, H, W)
    assert view.data_ptr() % 16
    for a, b in zip(grads(view), grads(view.clone())):
        assert torch.equal(a, b)
    one = torch.ones(1, device="cuda")
    for a, b in zip(grads(one.expand(3, H, W)), grads(torch.ones_like(hdr))):
        assert torch.equal(a, b)
