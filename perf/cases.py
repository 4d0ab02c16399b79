"""What this framework is measured on: the work its users have it do.

Kinds of work (``case["kind"]``), each through the package's public entry
points:

  frame       one frame of the plain method (``pipeline.Frame.run``): sample
              map, renderer stand-in, splat and pyramid, reconstruction with
              or without the temporal term, tone map
  sample_map  the sample-count map alone, in the modes a renderer picks
              (``Frame.alloc``, ``alloc_dithered``, ``alloc_systematic``)
  predict     one forward pass of the joint predictor (``learned.Predictor``)
  net_grad    a training step's network part: forward and backward of the
              joint predictor on a batch of crops
  train       a whole optimisation step of the predictor (``learned.Trainer``)
  two_stage   one frame of the sampler + denoiser pipeline
              (``two_stage.TwoStage``)
  recon_grad  the differentiable reconstruction under autograd
              (``autograd.Reconstruct`` and ``autograd.L1Loss``)
  conv_layer  one 3x3 convolution layer, forward, data gradient and weight
              gradient

Inputs are drawn on the device from the case's seed.  They follow the
repository's synthetic recipe: log-normal sampling density, piecewise
constant albedo under smooth light in [0, 4], unit-normal kernel logits, an
affine motion field of at most 8 pixels, about 5 % disoccluded pixels.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

import paper_2602_08642_gb300 as spp
from paper_2602_08642_gb300 import autograd, learned, two_stage
from paper_2602_08642_gb300.pipeline import logit_channels

B = spp.binding
DEV = "cuda"
PHI = 0.125       # uniform share of the sample budget
LAMBDA = 10.0     # slope of the holdout ramp
FEATURES = 12     # input channels of the joint predictor
# fine-tuning rate of the training case: a trained predictor adapted to a new
# scene, optimiser moments in hand
FINE_TUNE_LR = 1e-5


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest plain frame: a preview or a unit of an interactive tool,
        # single image, no history
        dict(name="frame_128", kind="frame", W=128, H=128, L=2, spp=0.25, temporal=False),
        # the standard real-time frame: full HD sequence with reprojection
        dict(name="frame_1080p", kind="frame", W=1920, H=1080, L=3, spp=0.25, temporal=True),
        # a laptop panel whose width is no multiple of four, at the low budget
        dict(name="frame_1366x768", kind="frame", W=1366, H=768, L=2, spp=0.125, temporal=True),
        # the largest display frame at the high budget
        dict(name="frame_4k", kind="frame", W=3840, H=2160, L=3, spp=0.5, temporal=True),
        # a renderer that takes its sample map from the library and must meet
        # the budget exactly on every frame
        dict(name="map_systematic_1440p", kind="sample_map", W=2560, H=1440, spp=0.25,
             mode="systematic"),
        # inference of the predictor for one full HD frame
        dict(name="predict_1080p", kind="predict", W=1920, H=1080, B=1),
        # and for one 4K frame, the largest call
        dict(name="predict_4k", kind="predict", W=3840, H=2160, B=1),
        # network forward and backward on a training batch
        dict(name="net_grad_8x256", kind="net_grad", W=256, H=256, B=8),
        # the whole optimisation step at the training configuration
        dict(name="train_8x256", kind="train", size=256, B=8, spp=0.25),
        # the two-network pipeline, one full HD frame of a running sequence
        dict(name="two_stage_1080p", kind="two_stage", W=1920, H=1080, spp=0.25),
        # a user's own training loop around the differentiable reconstruction
        dict(name="recon_grad_540p", kind="recon_grad", W=960, H=540, L=3, temporal=True),
        # a single hidden layer in a user's own network, ragged grid
        dict(name="conv_64_500x281", kind="conv_layer", W=500, H=281, B=2, cin=64, cout=64),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, lo, hi, mult):
    """W, H multiples of ``mult`` with lo^2 <= W H <= hi^2 in the logarithm
    and an aspect ratio between square and 2 : 1."""
    side = _log_uniform(rng, lo, hi)
    aspect = rng.uniform(1.0, 2.0)
    fit = lambda v: max(mult, int(v) // mult * mult)
    return fit(side * math.sqrt(aspect)), fit(side / math.sqrt(aspect))


def draw(rng):
    kind = rng.choice(["frame", "frame", "sample_map", "predict", "net_grad", "train", "two_stage",
                       "recon_grad", "conv_layer", "conv_layer"])
    if kind == "frame":
        L = rng.choice([2, 3, 3, 4, 5])
        W, H = _grid(rng, 64, 2700, 1 << (L - 1))
        return dict(kind=kind, W=W, H=H, L=L, spp=round(rng.uniform(0.11, 0.5), 3),
                    temporal=rng.random() < 0.7)
    if kind == "sample_map":
        W, H = _grid(rng, 64, 2800, 1)
        return dict(kind=kind, W=W, H=H, spp=round(_log_uniform(rng, 0.11, 4.0), 3),
                    mode=rng.choice(["ramp", "hard", "dithered", "systematic"]))
    if kind == "predict":
        W, H = _grid(rng, 64, 2000, 4)
        return dict(kind=kind, W=W, H=H, B=1 if W * H > 500000 else rng.choice([1, 2, 4]))
    if kind == "net_grad":
        W, H = _grid(rng, 32, 320, 4)
        return dict(kind=kind, W=W, H=H, B=rng.choice([1, 2, 4, 6]))
    if kind == "train":
        return dict(kind=kind, size=int(_log_uniform(rng, 48, 256)) // 4 * 4,
                    B=rng.choice([1, 2, 4, 6]), spp=round(rng.uniform(0.125, 0.5), 3))
    if kind == "two_stage":
        W, H = _grid(rng, 64, 1400, 4)
        return dict(kind=kind, W=W, H=H, spp=round(rng.uniform(0.125, 0.5), 3))
    if kind == "recon_grad":
        L = rng.choice([2, 3])
        W, H = _grid(rng, 32, 1000, 1 << (L - 1))
        return dict(kind=kind, W=W, H=H, L=L, temporal=rng.random() < 0.6)
    W, H = _grid(rng, 24, 500, 1)
    return dict(kind=kind, W=W, H=H, B=rng.choice([1, 2, 3]),
                cin=rng.choice([16, 32, 64, 96, 128]), cout=rng.choice([16, 32, 64, 96, 128]))


# ------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + 17)
    return g


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device=DEV) * (hi - lo) + lo


def _scene(g, W, H):
    """Clean radiance [3][H][W] in [0, 4] and the G-buffer of one frame:
    discs and half-planes of constant albedo and depth under smooth light."""
    ys, xs = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float32),
                            torch.arange(W, device=DEV, dtype=torch.float32), indexing="ij")
    label = torch.zeros(H, W, dtype=torch.int64, device=DEV)
    r = _uniform(g, 0.0, 1.0, 16, 5)
    for k in range(16):
        px, py, a, rad = r[k, 1] * W, r[k, 2] * H, r[k, 3] * 2 * math.pi, r[k, 4]
        if k % 2:
            inside = torch.cos(a) * (xs - px) + torch.sin(a) * (ys - py) > 0
        else:
            inside = (xs - px) ** 2 + (ys - py) ** 2 < ((0.05 + 0.2 * rad) * max(W, H)) ** 2
        label = torch.where(inside, k + 1, label)
    albedo = _uniform(g, 0.05, 1.0, 17, 3)[label].permute(2, 0, 1).contiguous()
    depth = _uniform(g, 1.0, 60.0, 17)[label]
    u, v = xs / max(W, H), ys / max(W, H)
    w = _uniform(g, 0.5, 4.0, 3, 3, 2)
    ph = _uniform(g, 0.0, 2 * math.pi, 3, 3)
    light = torch.stack([1 + sum(0.25 * torch.sin(2 * math.pi * (w[c, q, 0] * u + w[c, q, 1] * v)
                                                  + ph[c, q]) for q in range(3))
                         for c in range(3)])
    clean = (2.2 * albedo * light).clamp(0.0, 4.0).contiguous()
    bump = torch.sin(2 * math.pi * (w[0, 0, 0] * u + w[0, 0, 1] * v) + ph[0, 0])
    slope = torch.stack([0.4 * bump, 0.4 * bump.roll(1, 0), torch.ones_like(bump)])
    normal = (slope / slope.norm(dim=0, keepdim=True)).contiguous()
    depth = (depth + 0.3 * bump + 0.002 * (xs + ys)).clamp(1.0, 100.0)[None].contiguous()
    return clean, dict(albedo=albedo, normal=normal, depth=depth)


def _motion(g, W, H):
    """Affine motion field [2][H][W] of at most 8 pixels."""
    ys, xs = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float32) - (H - 1) / 2,
                            torch.arange(W, device=DEV, dtype=torch.float32) - (W - 1) / 2,
                            indexing="ij")
    A = _uniform(g, -1.0, 1.0, 2, 2) * (4.0 / max(W, H))
    b = _uniform(g, -4.0, 4.0, 2)
    mv = torch.stack([A[0, 0] * xs + A[0, 1] * ys + b[0], A[1, 0] * xs + A[1, 1] * ys + b[1]])
    return (mv * (8.0 / mv.norm(dim=0).max()).clamp(max=1.0)).contiguous()


def _mask(g, W, H):
    """Disoccluded pixels (uint8), discs over about 5 % of the frame."""
    ys, xs = torch.meshgrid(torch.arange(H, device=DEV), torch.arange(W, device=DEV),
                            indexing="ij")
    m = torch.zeros(H, W, dtype=torch.bool, device=DEV)
    rad = math.sqrt(0.05 * W * H / (math.pi * 24))
    p = _uniform(g, 0.0, 1.0, 24, 3)
    for k in range(24):
        m |= (xs - p[k, 0] * W) ** 2 + (ys - p[k, 1] * H) ** 2 < ((0.5 + p[k, 2]) * rad) ** 2
    return m.to(torch.uint8)


def _logits(g, W, H, L, temporal):
    return [torch.randn(logit_channels(l, L, temporal), H >> l, W >> l, generator=g, device=DEV)
            for l in range(L)]


def _density(g, W, H):
    return torch.randn(H, W, generator=g, device=DEV).exp()


def _theta(g, table, head_scale):
    """He-normal weights; heads scaled down, with the biases of the plain
    fixed kernels (denoise tap (i, j) gets -(i^2 + j^2) / 2)."""
    tap = torch.tensor([-(i * i + j * j) / 2.0 for j in range(-2, 3) for i in range(-2, 3)],
                       device=DEV)
    parts = []
    for name, cin, cout, relu in table:
        w = torch.randn(cout, cin, 3, 3, generator=g, device=DEV) * math.sqrt(2.0 / (9 * cin))
        b = torch.zeros(cout, device=DEV)
        if not relu:
            w *= head_scale
            if cout >= 25:
                b[:25] = tap
        parts += [w.reshape(-1), b]
    return torch.cat(parts)


def _features(g, W, H, batch):
    """The predictor's 12 input planes for a batch of frames."""
    out = torch.empty(batch, FEATURES, H, W, device=DEV)
    for b in range(batch):
        clean, gb = _scene(g, W, H)
        out[b, 0:3], out[b, 3:6] = gb["albedo"], gb["normal"]
        out[b, 6:7] = gb["depth"].log() / math.log(100.0)
        out[b, 7:9] = _motion(g, W, H) / 8
        out[b, 9:12] = (clean / 4).sqrt()
    return out


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    return _PREPARE[case["kind"]](case, _gen(seed))


def _prepare_frame(c, g):
    W, H, L, temporal = c["W"], c["H"], c["L"], c["temporal"]
    clean, _ = _scene(g, W, H)
    s = dict(c, d=_density(g, W, H), clean=clean, logits=_logits(g, W, H, L, temporal),
             frame=spp.Frame(W, H, L, max_budget=c["spp"]), prev=None, mv=None, mask=None)
    if temporal:
        s.update(prev=(clean * 0.8 + 0.2).contiguous(), mv=_motion(g, W, H), mask=_mask(g, W, H))
    return s


def _prepare_map(c, g):
    s = dict(c, d=_density(g, c["W"], c["H"]),
             frame=spp.Frame(c["W"], c["H"], 1, max_budget=c["spp"]))
    if c["mode"] == "dithered":
        mask = B.spp_blue_noise_mask(64, 11)
        s["mask"] = torch.from_numpy(mask.view("int16")).to(DEV)
    return s


def _prepare_net(c, g):
    grad = c["kind"] == "net_grad"
    theta = _theta(g, learned.layer_table(), 1.0)
    net = learned.Predictor(theta, c["B"], c["W"], c["H"], train=grad)
    net.in12.copy_(_features(g, c["W"], c["H"], c["B"]))
    if grad:
        n = c["B"] * c["W"] * c["H"]
        for t in net.g_logits:  # gradients of a mean over the batch's pixels
            t.copy_(torch.randn(t.shape, generator=g, device=DEV) / n)
    return dict(c, net=net, theta=theta)


def _prepare_train(c, g):
    S = c["size"]
    tr = learned.Trainer(_theta(g, learned.layer_table(), 0.1), c["B"], S, c["spp"],
                         lr=FINE_TUNE_LR)
    tr.net.m.copy_(torch.randn(tr.net.m.shape, generator=g, device=DEV) * 1e-4)
    tr.net.v.copy_(torch.randn(tr.net.v.shape, generator=g, device=DEV).exp() * 1e-6)
    tr.net.step_count = 1000
    samples = []
    for k in range(c["B"]):
        clean, gb = _scene(g, S, S)
        prev, gprev = clean.roll((1, -1), (1, 2)), {n: t.roll((1, -1), (1, 2))
                                                    for n, t in gb.items()}
        mv = torch.empty(2, S, S, device=DEV)
        mv[0], mv[1] = -1.0, 1.0
        host = lambda t: t.contiguous().cpu().numpy()
        samples.append(learned.FrameData(
            dict(clean=host(clean), clean_prev=host(prev), mv=host(mv),
                 gbuf={n: host(t) for n, t in gb.items()},
                 gbuf_prev={n: host(t) for n, t in gprev.items()}), seed=k))
    return dict(c, trainer=tr, samples=samples)


def _prepare_two_stage(c, g):
    W, H = c["W"], c["H"]
    th = [_theta(g, two_stage.layer_table(n), 0.1)
          for n in (B.SPP_NET_SAMPLER, B.SPP_NET_DENOISER)]
    p = two_stage.TwoStage(th[0], th[1], 1, W, H, c["spp"])
    clean, gb = _scene(g, W, H)
    s = dict(c, pipe=p, gbuf=gb, clean=clean, mv=_motion(g, W, H))
    p.begin_sequence()
    p.frame([gb], [s["mv"]], [clean], 5, 0)  # the sequence is running: history in hand
    return s


def _prepare_recon_grad(c, g):
    W, H, L, temporal = c["W"], c["H"], c["L"], c["temporal"]
    clean, _ = _scene(g, W, H)
    hits = (torch.rand(H, W, generator=g, device=DEV) < 0.25).float()
    layers = [(clean * hits * 4).contiguous()]
    for _ in range(1, L):
        layers.append(F.avg_pool2d(layers[-1][None], 2)[0].contiguous())
    leaf = lambda t: t.detach().requires_grad_(True)
    s = dict(c, layers=[leaf(t) for t in layers],
             logits=[leaf(t) for t in _logits(g, W, H, L, temporal)], warped=None, mask=None,
             ref=(clean / 4).sqrt(), tm=B.make_tonemap())
    if temporal:
        noise = torch.randn(3, H, W, generator=g, device=DEV) * 0.1
        s.update(warped=leaf((clean * noise.exp() + 0.01).contiguous()), mask=_mask(g, W, H))
    return s


def _prepare_conv(c, g):
    W, H, n, cin, cout = c["W"], c["H"], c["B"], c["cin"], c["cout"]
    bf = torch.bfloat16
    x = torch.randn(n, H, W, cin, generator=g, device=DEV).relu().to(bf)
    gy = (torch.randn(n, H, W, cout, generator=g, device=DEV) * 1e-3).to(bf)
    w = torch.randn(cout, cin, 3, 3, generator=g, device=DEV) * math.sqrt(2.0 / (9 * cin))
    u8 = lambda k: torch.empty(max(int(k), 16), dtype=torch.uint8, device=DEV)
    return dict(c, x=x, gy=gy, w=w, bias=torch.randn(cout, generator=g, device=DEV) * 0.1,
                y=torch.empty(n, H, W, cout, dtype=bf, device=DEV), gx=torch.empty_like(x),
                gw=torch.empty_like(w), gb=torch.empty(cout, device=DEV),
                ws=u8(B.spp_conv3x3_workspace_bytes(cin, cout)),
                wws=u8(B.spp_conv3x3_backward_weights_workspace_bytes(n, W, H, cin, cout)),
                status=torch.zeros(4, dtype=torch.int32, device=DEV)[:1])


_PREPARE = dict(frame=_prepare_frame, sample_map=_prepare_map, predict=_prepare_net,
                net_grad=_prepare_net, train=_prepare_train, two_stage=_prepare_two_stage,
                recon_grad=_prepare_recon_grad, conv_layer=_prepare_conv)


# ---------------------------------------------------------------------- run
def run(s):
    return _RUN[s["kind"]](s)


def _run_frame(s):
    fr = s["frame"]
    hdr = fr.run(s["d"], s["clean"], s["logits"], B.make_params(s["spp"], seed=7, frame=3),
                 prev=s["prev"], mv=s["mv"], mask=s["mask"])
    return dict(hdr=hdr, ldr=fr.ldr, counts=fr.counts, offsets=fr.offsets, s=fr.s,
                holdout_w=fr.holdout_w, layers=fr.layers)


def _run_map(s):
    fr, mode = s["frame"], s["mode"]
    p = B.make_params(s["spp"], seed=7, frame=3, hard=mode == "hard")
    if mode == "systematic":
        fr.alloc_systematic(s["d"], p)
    elif mode == "dithered":
        fr.alloc_dithered(s["d"], p, s["mask"])
    else:
        fr.alloc(s["d"], p)
    return dict(counts=fr.counts, offsets=fr.offsets, s=fr.s, holdout_w=fr.holdout_w,
                total=fr.total)


def _run_predict(s):
    net = s["net"]
    net.forward()
    return dict(density=net.density, logits=net.logits)


def _run_net_grad(s):
    net = s["net"]
    net.forward()
    net.backward()
    return dict(logits=net.logits, grad=net.grad)


def _run_train(s):
    tr = s["trainer"]
    loss = tr.step(s["samples"], 40)
    net = tr.net
    return dict(loss=loss, theta=net.theta, grad=net.grad, m=net.m, v=net.v, density=net.density,
                ldr=tr.rnd.ldr)


def _run_two_stage(s):
    p = s["pipe"]
    p.frame([s["gbuf"]], [s["mv"]], [s["clean"]], 5, 1)
    return dict(hdr=p.hdr[0], ldr=p.ldr[0], density=p.sampler.density, counts=p.frames[0].counts,
                latent=p.latent[0], m=p.m[0])


def _run_recon_grad(s):
    L = s["L"]
    hdr, ldr = autograd.Reconstruct.apply(L, s["tm"], s["warped"], s["mask"], *s["layers"],
                                          *s["logits"])
    loss = autograd.L1Loss.apply(ldr, s["ref"])
    inputs = s["layers"] + s["logits"] + ([s["warped"]] if s["temporal"] else [])
    return dict(hdr=hdr.detach(), ldr=ldr.detach(), loss=loss.detach(),
                grads=list(torch.autograd.grad(loss, inputs)))


def _run_conv(s):
    W, H, n, cin, cout = s["W"], s["H"], s["B"], s["cin"], s["cout"]
    B.check(B.spp_conv3x3_forward(s["x"], n, W, H, cin, cout, s["w"], s["bias"], True, s["y"],
                                  s["ws"], s["status"]), "forward")
    B.check(B.spp_conv3x3_backward_data(s["gy"], n, W, H, cin, cout, s["w"], s["x"], s["gx"],
                                        s["ws"], s["status"]), "data gradient")
    B.check(B.spp_conv3x3_backward_weights(s["x"], s["gy"], n, W, H, cin, cout, s["gw"], s["gb"],
                                           s["wws"], s["status"]), "weight gradient")
    return dict(y=s["y"], gx=s["gx"], gw=s["gw"], gb=s["gb"])


_RUN = dict(frame=_run_frame, sample_map=_run_map, predict=_run_predict, net_grad=_run_net_grad,
            train=_run_train, two_stage=_run_two_stage, recon_grad=_run_recon_grad,
            conv_layer=_run_conv)


# --------------------------------------------------------------------- work
def _trunk(cin, h0, h1, h2):
    """(cin, cout, level) of a network's layers."""
    return [(cin, 32, 0), (32, 32, 0), (32, 64, 1), (64, 64, 1), (64, 128, 2), (128, 128, 2),
            (128, h2, 2), (192, 64, 1), (64, 64, 1), (64, h1, 1), (96, 32, 0), (32, 32, 0),
            (32, h0, 0)]


def _net_flops(layers, n):
    return sum(2.0 * 9 * ci * co * n / 4 ** l for ci, co, l in layers)


def _frame_bytes(n, L, spp_, temporal):
    lower = sum(4.0 ** -l for l in range(1, L))
    logits = sum(4 * logit_channels(l, L, temporal) * n / 4 ** l for l in range(L))
    # density, clean samples, logits and history in; counts, offsets, s, the
    # holdout weight, layers, HDR and sRGB out
    b = 4 * n + 12 * n * min(spp_, 1.0) + logits + 16 * n + 12 * n * (1 + lower) + 24 * n
    return b + (12 + 8 + 1) * n if temporal else b


def work(case):
    c, k = case, case["kind"]
    n = (c["size"] ** 2 if k == "train" else c["W"] * c["H"]) * c.get("B", 1)
    joint = _trunk(FEATURES, 55, 29, 25)
    heads = 4.0 * (55 + 29 / 4 + 25 / 16)  # bytes of logits per pixel
    params = 535565
    if k == "frame":
        taps = 54 if c["temporal"] else 29
        return dict(bytes=_frame_bytes(n, c["L"], c["spp"], c["temporal"]),
                    flops=8.0 * n * (taps + 29 / 3) + 200.0 * n)
    if k == "sample_map":
        return dict(bytes=20.0 * n + 4 * c["spp"] * n, flops=40.0 * n)
    if k == "predict":
        return dict(bytes=n * (4 * FEATURES + heads + 4) + 2.0 * params,
                    flops=_net_flops(joint, n))
    if k == "net_grad":
        return dict(bytes=n * (4 * FEATURES + 2 * heads) + 6.0 * params,
                    flops=3 * _net_flops(joint, n) - _net_flops(joint[:1], n))
    if k == "train":
        # two forward passes (frames t - 1 and t), one backward, the frames'
        # reconstruction, optimiser state in and out
        return dict(bytes=2.0 * _frame_bytes(n, 3, c["spp"], True) + n * 2 * heads + 28.0 * params,
                    flops=4 * _net_flops(joint, n) + 3000.0 * n)
    if k == "two_stage":
        nets = _net_flops(_trunk(19, 1, 0, 0), n) + _net_flops(_trunk(24, 64, 29, 25), n)
        # G-buffer, motion, clean samples and history in; HDR, sRGB, latents out
        return dict(bytes=n * (28.0 + 8 + 12 * c["spp"] + 12 + 28 + 24 + 28 + 20), flops=nets)
    if k == "recon_grad":
        lower = sum(4.0 ** -l for l in range(c["L"]))
        lg = sum(4.0 * logit_channels(l, c["L"], c["temporal"]) / 4 ** l for l in range(c["L"]))
        t = 24.0 if c["temporal"] else 0.0
        return dict(bytes=n * (2 * lg + 24 * lower + t + 12 + 24),
                    flops=30.0 * n * (54 if c["temporal"] else 29))
    return dict(bytes=n * 4.0 * (c["cin"] + c["cout"]) + 8.0 * 9 * c["cin"] * c["cout"],
                flops=3 * 2.0 * 9 * c["cin"] * c["cout"] * n)


# -------------------------------------------------------------------- exact
# The same results in 64 bits, from the definitions, on plain torch tensors.
def exact(case, seed):
    f = _EXACT.get(case["kind"])
    return f(case, prepare(case, seed)) if f else None


_GAMMA = -7046029254386353131     # 0x9E3779B97F4A7C15 as a signed word
_MUL1 = -4658895280553007687      # 0xBF58476D1CE4E5B9
_MUL2 = -7723592293110705685      # 0x94D049BB133111EB
_WORD = (1 << 64) - 1


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _mix(z):
    """SplitMix64's output function on signed 64-bit words."""
    z = (z ^ _shr(z, 30)) * _MUL1
    z = (z ^ _shr(z, 27)) * _MUL2
    return z ^ _shr(z, 31)


def _key(seed, frame):
    z = (seed + (frame + 1) * (_GAMMA & _WORD)) & _WORD
    z = ((z ^ (z >> 30)) * (_MUL1 & _WORD)) & _WORD
    z = ((z ^ (z >> 27)) * (_MUL2 & _WORD)) & _WORD
    z ^= z >> 31
    return z - (1 << 64) if z >= 1 << 63 else z


def _bits(key, i):
    return _mix(i * _GAMMA + _GAMMA + key)


def _exact_density(d, budget):
    """s = phi B + (1 - phi) B N d / sum d with the sum exact, each operation
    rounded once."""
    d = d.reshape(-1).double()
    total = math.fsum(d.tolist())
    return d * (((1.0 - PHI) * budget * d.numel()) / total) + PHI * budget


def _offsets(counts):
    zero = torch.zeros(1, dtype=torch.int64, device=DEV)
    return torch.cat([zero, counts.cumsum(0)]).to(torch.int32)


def _exact_map(c, s):
    """(counts, offsets, s, holdout weight) in 64 bits."""
    sd = _exact_density(s["d"], c["spp"])
    n = sd.numel()
    i = torch.arange(n, device=DEV)
    h = 2 * LAMBDA / (2 * LAMBDA - 1)
    hard = c.get("mode") == "hard"
    if c.get("mode") == "systematic":
        q = (sd * 2.0 ** 32).round().to(torch.int64)
        U = _shr(_bits(_key(7, 3), torch.tensor([1 << 62], device=DEV)), 32)
        ends = torch.cat([U, U + q.cumsum(0)])
        offsets, counts = (ends >> 32).to(torch.int32), (ends[1:] >> 32) - (ends[:-1] >> 32)
        u = (ends[:-1] & 0xFFFFFFFF).double() * 2.0 ** -32
        p = (q & 0xFFFFFFFF).double() * 2.0 ** -32
        extra = u + p >= 1.0
    else:
        if c.get("mode") == "dithered":
            T = s["mask"].shape[0]
            rank = (s["mask"].to(torch.int64) & 0xFFFF)[(i // c["W"]) % T, (i % c["W"]) % T]
            k = 2 * int(math.log2(T))
            z = torch.tensor([7], device=DEV)
            off = (3 * ((_GAMMA & _WORD) >> 16) + int(_shr(_mix(z), 16))) & ((1 << 48) - 1)
            u = (rank * (1 << (48 - k)) + (1 << (47 - k)) + off) & ((1 << 48) - 1)
        else:
            u = _shr(_bits(_key(7, 3), i), 16)
        u = u.double() * 2.0 ** -48
        f = sd.floor()
        p = sd - f
        extra = (p > 0) & (u > 1.0 - p)
        counts = f.to(torch.int64) + extra
        offsets = _offsets(counts)
    w = h * ((LAMBDA / p.clamp(min=1e-300)) * (u + p - 1.0)).clamp(0.0, 1.0)
    w = torch.where(extra, w, 1.0) if not hard else torch.ones_like(sd)
    return counts, offsets, sd, w


def _exact_sample_map(c, s):
    counts, offsets, sd, w = _exact_map(c, s)
    return dict(counts=counts.to(torch.int32), offsets=offsets, s=sd, holdout_w=w,
                total=offsets[-1:].to(torch.int64))


def _render(clean, key, pixel, slot):
    """Samples [n][3]: clean radiance times exp(0.8 Z - 0.32), Z normal."""
    hp = _bits(key, pixel)
    u1 = (_shr(_mix(hp + (2 * slot + 1) * _GAMMA), 40).double() + 0.5) * 2.0 ** -24
    u2 = _shr(_mix(hp + (2 * slot + 2) * _GAMMA), 40).double() * 2.0 ** -24
    z = torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2 * math.pi * u2)
    return clean.reshape(3, -1).double()[:, pixel].T * torch.exp(0.8 * z - 0.32)[:, None]


def _warp(prev, mv):
    _, H, W = prev.shape
    ys, xs = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float64),
                            torch.arange(W, device=DEV, dtype=torch.float64), indexing="ij")
    x = (xs + mv[0].double()).clamp(0, W - 1)
    y = (ys + mv[1].double()).clamp(0, H - 1)
    x0, y0 = x.floor(), y.floor()
    fx, fy = x - x0, y - y0
    x0, y0 = x0.long(), y0.long()
    x1, y1 = (x0 + 1).clamp(max=W - 1), (y0 + 1).clamp(max=H - 1)
    P = prev.double()
    return ((1 - fy) * ((1 - fx) * P[:, y0, x0] + fx * P[:, y0, x1])
            + fy * ((1 - fx) * P[:, y1, x0] + fx * P[:, y1, x1]))


def _level(noisy, logits, coarse, warped, mask):
    """One level of the gather pyramid: joint softmax of the kernels present,
    5x5 taps with clamped borders, 2x2 upsampling taps at floor((x + i) / 2)."""
    _, H, W = noisy.shape
    ys, xs = torch.arange(H, device=DEV), torch.arange(W, device=DEV)

    def taps(img, n):
        for k in range(n):
            if n == 25:
                yy, xx = (ys + k // 5 - 2).clamp(0, H - 1), (xs + k % 5 - 2).clamp(0, W - 1)
            else:
                yy = ((ys + k // 2) // 2).clamp(max=H // 2 - 1)
                xx = ((xs + k % 2) // 2).clamp(max=W // 2 - 1)
            yield k, img.index_select(1, yy).index_select(2, xx)

    groups = [(0, 25, noisy)]
    if coarse is not None:
        groups.append((25, 4, coarse))
    if warped is not None:
        groups.append((29, 25, warped))
    live = logits.double()[:groups[-1][0] + groups[-1][1]]
    if warped is not None:
        off = torch.zeros_like(live, dtype=torch.bool)
        off[29:] = mask.bool()
        live = live.masked_fill(off, -math.inf)
    weight = torch.softmax(live, 0)
    out = 0.0
    for first, n, img in groups:
        for k, v in taps(img.double(), n):
            out = out + weight[first + k] * v
    return out


def _tonemap(hdr):
    """The default tone map (unit contrast and saturation, zero exposure,
    shadow and highlight 1/2) and the sRGB encoding."""
    x = hdr.clamp(min=2.0 ** -24).log()
    toe, shoulder = 0.25 * torch.exp((x + 0.5) / 0.5), 1 - 0.25 * torch.exp(-(x - 0.5) / 0.5)
    v = torch.where(x < -0.5, toe, torch.where(x < 0.5, 0.5 * (1 + x), shoulder))
    return torch.where(v <= 0.0031308, 12.92 * v,
                       1.055 * v.clamp(min=0.0031308) ** (1 / 2.4) - 0.055)


def _reconstruct(layers, logits, warped, mask):
    hat = None
    for l in range(len(layers) - 1, -1, -1):
        hat = _level(layers[l], logits[l], hat, warped if l == 0 else None, mask)
    return hat


def _exact_frame(c, s):
    W, H = c["W"], c["H"]
    counts, offsets, sd, w = _exact_map(c, s)
    n = sd.numel()
    pixel = torch.repeat_interleave(torch.arange(n, device=DEV), counts)
    slot = torch.arange(pixel.numel(), device=DEV) - offsets[:-1].long()[pixel]
    rgb = _render(s["clean"], _key(0xC0FFEE, 3), pixel, slot)
    rgb = torch.where((slot == counts[pixel] - 1)[:, None], rgb * w[pixel][:, None], rgb)
    total = torch.zeros(n, 3, dtype=torch.float64, device=DEV).index_add_(0, pixel, rgb)
    layers = [(total / sd[:, None]).T.reshape(3, H, W)]
    for _ in range(1, c["L"]):
        layers.append(F.avg_pool2d(layers[-1][None], 2)[0])
    warped = _warp(s["prev"], s["mv"]) if c["temporal"] else None
    hdr = _reconstruct(layers, s["logits"], warped, s["mask"])
    return dict(hdr=hdr, ldr=_tonemap(hdr), counts=counts.to(torch.int32), offsets=offsets, s=sd,
                holdout_w=w, layers=layers)


def _exact_recon_grad(c, s):
    leaf = lambda t: t.detach().double().requires_grad_(True)
    layers, logits = [leaf(t) for t in s["layers"]], [leaf(t) for t in s["logits"]]
    warped = leaf(s["warped"]) if c["temporal"] else None
    hdr = _reconstruct(layers, logits, warped, s["mask"])
    ldr = _tonemap(hdr)
    loss = (ldr - s["ref"].double()).abs().mean()
    grads = torch.autograd.grad(loss, layers + logits + ([warped] if c["temporal"] else []))
    return dict(hdr=hdr.detach(), ldr=ldr.detach(), loss=loss.detach(), grads=list(grads))


def _conv64(x, w, b, rows=64):
    """3x3 convolution in 64 bits, a band of rows at a time (one matrix
    product per tap)."""
    n, cin, H, W = x.shape
    x = F.pad(x, (1, 1, 1, 1))
    out = torch.empty(n, w.shape[0], H, W, dtype=torch.float64, device=DEV)
    for i in range(n):
        for y in range(0, H, rows):
            h = min(rows, H - y)
            acc = b[:, None]
            for t in range(9):
                win = x[i, :, y + t // 3:y + t // 3 + h, t % 3:t % 3 + W].reshape(cin, -1)
                acc = acc + w[:, :, t // 3, t % 3] @ win
            out[i, :, y:y + h] = acc.reshape(-1, h, W)
    return out


def _exact_predict(c, s):
    if c["W"] * c["H"] * c["B"] > 2200000:
        return None  # minutes in 64 bits
    x, at, layer = s["net"].in12.double(), 0, {}
    for name, cin, cout, relu in learned.layer_table():
        w = s["theta"][at:at + cout * cin * 9].double().reshape(cout, cin, 3, 3)
        at += cout * cin * 9
        layer[name] = (w, s["theta"][at:at + cout].double(), relu)
        at += cout

    def conv(name, x):
        w, b, relu = layer[name]
        y = _conv64(x, w, b)
        return y.relu_() if relu else y

    up = lambda x: x.repeat_interleave(2, 2).repeat_interleave(2, 3)
    s0 = conv("e0b", conv("e0a", x))
    s1 = conv("e1b", conv("e1a", F.avg_pool2d(s0, 2)))
    bt = conv("e2b", conv("e2a", F.avg_pool2d(s1, 2)))
    t1 = conv("d1b", conv("d1a", torch.cat([s1, up(bt)], 1)))
    t0 = conv("d0b", conv("d0a", torch.cat([s0, up(t1)], 1)))
    h0 = conv("h0", t0)
    z = h0[:, 54]
    return dict(density=torch.exp(z - z.amax((1, 2), keepdim=True)),
                logits=[h0, conv("h1", t1), conv("h2", bt)])


def _exact_net_grad(c, s):
    # the parameter gradients have no value beyond about 10 %: BF16 decides
    # which pre-activations near zero the ReLU passes
    p = _exact_predict(c, s)
    return p and dict(logits=p["logits"], grad=None)


def _exact_conv(c, s):
    cin, cout = c["cin"], c["cout"]
    # the layer's precision is that of its operands: BF16 weights
    w = s["w"].to(torch.bfloat16).double()
    x, gy = (s[k].double().permute(0, 3, 1, 2) for k in ("x", "gy"))
    y = _conv64(x, w, s["bias"].double()).relu()
    gx = _conv64(gy, w.flip(2, 3).transpose(0, 1).contiguous(),
                 torch.zeros(cin, dtype=torch.float64, device=DEV))
    gx = torch.where(x > 0, gx, 0.0)
    xp = F.pad(x, (1, 1, 1, 1))
    H, W = c["H"], c["W"]
    gw = torch.empty(cout, cin, 3, 3, dtype=torch.float64, device=DEV)
    flat = gy.permute(1, 0, 2, 3).reshape(cout, -1)
    for t in range(9):
        win = xp[:, :, t // 3:t // 3 + H, t % 3:t % 3 + W].permute(1, 0, 2, 3).reshape(cin, -1)
        gw[:, :, t // 3, t % 3] = flat @ win.T
    nhwc = lambda t: t.permute(0, 2, 3, 1).contiguous()
    return dict(y=nhwc(y), gx=nhwc(gx), gw=gw, gb=flat.sum(1))


_EXACT = dict(frame=_exact_frame, sample_map=_exact_sample_map, predict=_exact_predict,
              net_grad=_exact_net_grad, recon_grad=_exact_recon_grad, conv_layer=_exact_conv)
