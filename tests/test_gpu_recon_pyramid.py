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


def test_ldr_gradient_views_of_any_alignment(spp):
    """The same for the tone-mapped output, alone and joined to the HDR one by a
    concatenation, whose backward hands out such views."""
    from paper_2602_08642_gb300 import autograd
    W, H, L = 30, 6, 2  # 3 W H is no multiple of 8
    g = torch.Generator(device="cuda").manual_seed(6)
    leaf = lambda *s: torch.randn(*s, generator=g, device="cuda").requires_grad_(True)
    layers = [leaf(3, H >> l, W >> l) for l in range(L)]
    logits = [leaf(29, H, W), leaf(25, H // 2, W // 2)]
    hdr, ldr = autograd.Reconstruct.apply(L, spp.binding.make_tonemap(), None, None, *layers, *logits)
    inputs = layers + logits
    grads = lambda go: torch.autograd.grad(ldr, inputs, go, retain_graph=True)
    buf = torch.randn(3 * H * W + 1, generator=g, device="cuda")
    view = buf[1:].view(3, H, W)
    assert view.data_ptr() % 16
    for a, b in zip(grads(view), grads(view.clone())):
        assert torch.equal(a, b)
    n = 3 * H * W
    both = torch.randn(2 * n + 1, generator=g, device="cuda")
    cat = torch.cat([torch.zeros(1, device="cuda"), ldr.flatten(), hdr.flatten()])
    got = torch.autograd.grad(cat, inputs, both, retain_graph=True)
    want = torch.autograd.grad([ldr, hdr], inputs, [both[1:n + 1].view_as(ldr).clone(),
                                                    both[n + 1:].view_as(hdr).clone()])
    for a, b in zip(got, want):
        assert torch.equal(a, b)


def test_gradient_views_of_any_alignment_elsewhere(spp):
    """The warp, the splat and the density take such views too, and transposed ones.
    The warp's backward adds with atomics: FP32 rounding of its few terms, 1e-5."""
    from paper_2602_08642_gb300 import autograd
    W, H, L = 36, 12, 2
    g = torch.Generator(device="cuda").manual_seed(7)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")

    def views(*shape):
        """The same values as a plain tensor, from an odd offset, and transposed."""
        plain = rnd(*shape)
        buf = torch.zeros(plain.numel() + 1, device="cuda")
        buf[1:] = plain.flatten()
        odd = buf[1:].view(shape)
        assert odd.data_ptr() % 16
        return plain, odd, plain.transpose(-1, -2).contiguous().transpose(-1, -2)

    prev = rnd(3, H, W).requires_grad_(True)
    out = autograd.WarpPrevious.apply(prev, rnd(2, H, W))
    got = [torch.autograd.grad(out, prev, v, retain_graph=True)[0] for v in views(3, H, W)]
    assert all(torch.allclose(a, got[0], rtol=1e-5, atol=1e-5) for a in got)

    fr = spp.Frame(W, H, L, max_budget=1.0)
    params = spp.make_params(1.0, frame=1)
    z = rnd(H, W)
    d = (z - z.max()).exp()
    fr.alloc(d, params)
    fr.render(rnd(3, H, W).exp(), 5, 1)
    fr.splat()
    s = fr.s.clone().requires_grad_(True)
    layers = autograd.Splat.apply(fr, params, s)
    got = [torch.autograd.grad(layers, s, gs, retain_graph=True)[0]
           for gs in zip(views(3, H, W), views(3, H // 2, W // 2))]
    assert all(torch.equal(a, got[0]) for a in got)
    zt = z.requires_grad_(True)
    sz = autograd.DensityToS.apply(d, fr.s, 1.0, 0.125, zt)
    got = [torch.autograd.grad(sz, zt, v, retain_graph=True)[0] for v in views(H, W)]
    assert all(torch.equal(a, got[0]) for a in got)
