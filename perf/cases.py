"""The calls that users of this framework make, at the sizes they make them:
what `perf` measurements time and compare.

A case is a dict of plain values; `prepare` makes its inputs on the GPU from
a seed together with the plan, weights or table that a program keeps,
`run` makes one pass through the public entry points, and `exact` gives the
same outputs from plain torch in float64.  Eight kinds of call:

  render   one scene rendered (Renderer.render)
  batch    scenes with uneven particle counts rendered at once (Renderer.batch)
  adjoint  a render and its adjoint, as one step of inverse rendering makes
           them (Renderer.render_keep, Renderer.backward_kept)
  loss     the image losses of inverse rendering and their gradient
           (inverse.ImageLoss)
  noise    sensor noise on rendered images (noise.sensor_noise)
  conv     one convolution layer of the warm-start network, forward, data
           gradient and filter gradient (cnn.conv2d and its two adjoints)
  net      the whole network, forward and backward (cnn.WarmStartNet)
  infer    the whole network, forward only, on full images
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2606_21381_gb300 import cnn, inverse, noise, scenes
from paper_2606_21381_gb300.render import Renderer

BF, OBLIQUE, DIC = scenes.MODE_BF, scenes.MODE_OBLIQUE, scenes.MODE_DIC
OPTICS_GRADS = ("defocus", "shear_px", "shear_angle", "bias_phase")


def listed():
    return [
        # the plain image: a small canvas, where launches and latency count
        dict(name="render_256", kind="render", H=256, W=256, n=64, modes=BF | OBLIQUE, NA=0.4,
             defocus=0.0, mu=0.0, scale=1.0),
        # a rectangular field of view with every modality, out of focus, an
        # odd number of absorbing particles
        dict(name="render_512x1024_all_modes", kind="render", H=512, W=1024, n=1501,
             modes=BF | OBLIQUE | DIC, NA=0.5, defocus=1.3, mu=0.02, scale=1.0),
        # the largest single scene: 40,000 particles on 2048 x 2048
        dict(name="render_2048_40k", kind="render", H=2048, W=2048, n=40000, modes=OBLIQUE,
             NA=0.4, defocus=0.0, mu=0.02, scale=1.0),
        # a batch of heavily overlapping DIC images, each at its own defocus
        dict(name="batch_dic_1024", kind="batch", S=16, size=1024, lo=4000, hi=4000, modes=DIC,
             NA=0.5, defocus=2.0, mu=0.0, scale=1.8),
        # the batched workload: 32 scenes of 1,000 to 40,000 particles
        dict(name="batch_2048", kind="batch", S=32, size=2048, lo=1000, hi=40000, modes=OBLIQUE,
             NA=0.4, defocus=0.0, mu=0.02, scale=1.0),
        # one step of inverse rendering on the 512 x 512 scene
        dict(name="adjoint_512", kind="adjoint", H=512, W=512, n=200, modes=BF | DIC, NA=0.4,
             defocus=0.4, mu=0.02, scale=1.0),
        # the same on a dense DIC image of the 1024 x 1024 batch
        dict(name="adjoint_1024_dic", kind="adjoint", H=1024, W=1024, n=4000, modes=DIC, NA=0.5,
             defocus=-1.1, mu=0.0, scale=1.8),
        # both image losses of an inverse-rendering step, with the gradient
        dict(name="loss_512", kind="loss", K=2, H=512, W=512, cut_na=0.3, spectral=1e-3),
        # sensor noise on a batch of images at a camera's usual exposure
        dict(name="noise_16x1024", kind="noise", S=16, H=1024, W=1024, photons=1000.0, sigma=1.5),
        # the widest layer of the network on a training batch of 64 crops
        dict(name="conv_128_128", kind="conv", N=64, H=32, W=32, C=128, K=128, R=3, stride=1),
        # a strided layer whose sizes divide by nothing
        dict(name="conv_40_72_ragged", kind="conv", N=33, H=63, W=61, C=40, K=72, R=3, stride=2),
        # a training step's network pass on 64 crops of 256 x 256
        dict(name="net_64x256", kind="net", N=64, H=256, W=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One case of the listed ones' ranges."""
    kind = rng.choice(["render", "render", "batch", "batch", "adjoint", "adjoint", "loss",
                       "noise", "conv", "conv", "conv", "net", "infer"])
    modes = rng.choice([BF, OBLIQUE, DIC, BF | OBLIQUE, BF | DIC, BF | OBLIQUE | DIC])
    optics = dict(modes=modes, NA=round(rng.uniform(0.3, 0.6), 3),
                  defocus=rng.choice([0.0, round(rng.uniform(-2.0, 2.0), 3)]),
                  mu=rng.choice([0.0, 0.02]), scale=rng.choice([1.0, 1.8]))
    if kind in ("render", "adjoint"):
        top = 11 if kind == "render" else 10
        H, W = 2 ** rng.randint(7, top), 2 ** rng.randint(7, top)
        most = min(40000 if kind == "render" else 4000, H * W // 100)
        return dict(kind=kind, H=H, W=W, n=_log_int(rng, 16, most), **optics)
    if kind == "batch":
        size = 2 ** rng.randint(8, 11)
        K = bin(modes).count("1")
        S = _log_int(rng, 2, min(48, 32 * 2048 * 2048 // (size * size * K)))
        hi = size * size // 110
        return dict(kind=kind, S=S, size=size, lo=max(8, hi // rng.choice([4, 16, 40])), hi=hi,
                    **optics)
    if kind == "loss":
        return dict(kind=kind, K=rng.randint(1, 3), H=2 ** rng.randint(7, 11),
                    W=2 ** rng.randint(7, 11), cut_na=round(rng.uniform(0.1, 0.5), 4),
                    spectral=rng.choice([0.0, 1e-3]))
    if kind == "noise":
        return dict(kind=kind, S=rng.randint(1, 16), H=_log_int(rng, 100, 1024),
                    W=_log_int(rng, 100, 1024), photons=round(math.exp(rng.uniform(1.0, 10.0)), 2),
                    sigma=rng.choice([0.0, round(rng.uniform(0.5, 5.0), 2)]))
    if kind == "conv":
        # as wide as the image allows at the work of the largest layer
        H, W = _log_int(rng, 9, 130), _log_int(rng, 9, 130)
        C, K, R = 8 * _log_int(rng, 1, 16), 8 * _log_int(rng, 1, 16), rng.choice([1, 3, 3, 3, 5])
        stride = rng.choice([1, 1, 2])
        N = max(1, min(64, 64 * 32 * 32 * 128 * 128 * 9 * stride ** 2 // (H * W * C * K * R * R),
                       2 ** 26 // (H * W * max(C, K))))
        return dict(kind=kind, N=_log_int(rng, 1, N), H=H, W=W, C=C, K=K, R=R, stride=stride)
    H, W = 8 * _log_int(rng, 6, 64), 8 * _log_int(rng, 6, 64)
    return dict(kind=kind, N=_log_int(rng, 1, max(1, min(64, 64 * 256 * 256 // (H * W)))), H=H,
                W=W)


# ------------------------------------------------------------------ inputs
def _scene(rng, n, H, W, case):
    mu = (0.005, case["mu"]) if case["mu"] > 0 else (0.0, 0.0)
    return scenes.draw_particles(rng, n, H, W, dn=(0.005, 0.06), mu=mu,
                                 size_scale=case["scale"])


def _optics(rng, H, W, case):
    o = scenes.optics(H, W, modes=case["modes"], NA=case["NA"], defocus=case["defocus"])
    o["oblique_angle"] = float(rng.uniform(0.0, 2.0 * math.pi))
    return o


def _batch_scenes(case, seed):
    rng = np.random.default_rng(seed)
    S, size = case["S"], case["size"]
    n = [int(round(math.exp(v))) for v in rng.uniform(math.log(case["lo"]),
                                                       math.log(case["hi"]), S - 1)]
    n.append(case["hi"])
    rng.shuffle(n)
    soas = [_scene(rng, k, size, size, case) for k in n]
    optics = [_optics(rng, size, size, case) for _ in n]
    if case["defocus"]:
        for o in optics:
            o["defocus"] = float(rng.uniform(-1.0, 1.0)) * case["defocus"]
    return soas, optics


def _normal(gen, shape, dev, scale=1.0):
    return (torch.randn(shape, generator=gen) * scale).to(dev)


def _smooth_images(gen, shape, dev):
    """Images like rendered ones, around 1, with bright and dark spots of a
    few pixels and a few pixels without any light."""
    *lead, H, W = shape
    n = int(np.prod(lead)) if lead else 1
    low = torch.randn((n, 1, max(2, H // 8), max(2, W // 8)), generator=gen).to(dev)
    field = F.interpolate(low, size=(H, W), mode="bilinear", align_corners=False)
    return (1.0 + 0.5 * field).clamp_(min=0.0).reshape(shape).contiguous()


def _conv_tensors(case, seed, dev):
    N, H, W, C, K, R, st = (case[k] for k in ("N", "H", "W", "C", "K", "R", "stride"))
    gen = torch.Generator(device=dev).manual_seed(seed)
    rand = lambda *s: torch.randn(s, generator=gen, device=dev)  # noqa: E731
    P, Q = (H + 2 * (R // 2) - R) // st + 1, (W + 2 * (R // 2) - R) // st + 1
    x = rand(N, H, W, C).clamp_(min=0.0).to(torch.bfloat16)  # what a ReLU passes on
    w = (rand(K, R, R, C) * math.sqrt(2.0 / (R * R * C))).to(torch.bfloat16)
    b = rand(K) * 0.1
    dy = (rand(N, P, Q, K) * 1e-2).to(torch.bfloat16)
    return x, w, b, dy


def _net_tensors(case, seed, dev):
    N, H, W = case["N"], case["H"], case["W"]
    gen = torch.Generator().manual_seed(seed)
    w, b = [], []
    for cin, cout, k, _, _ in _net_specs():
        fan = k * k * (2 if cin == cnn.IN_CHANNELS else cin)
        w.append(_normal(gen, (cout, k, k, cin), dev, math.sqrt(2.0 / fan)))
        b.append(_normal(gen, (cout,), dev, 0.05))
    g = torch.Generator(device=dev).manual_seed(seed)
    images = 1.0 + 0.3 * torch.randn((N, 2, H, W), generator=g, device=dev)
    x = torch.zeros((N, H, W, cnn.IN_CHANNELS), dtype=torch.bfloat16, device=dev)
    x[..., :2] = 2.0 * (images - images.mean(dim=(2, 3), keepdim=True)).permute(0, 2, 3, 1)
    h, v = H, W
    for _, _, k, st, pad in _net_specs():
        h, v = (h + 2 * pad - k) // st + 1, (v + 2 * pad - k) // st + 1
    dout = torch.randn((N, h, v, cnn.OUT_CHANNELS), generator=g, device=dev) * 1e-2
    return w, b, x, dout


def _net_specs():
    specs = [(cin, cout, 3, st, 1) for cin, cout, st in cnn.LAYERS]
    return specs + [(cnn.LAYERS[-1][1], cnn.OUT_CHANNELS, 1, 1, 0)]


def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind in ("render", "adjoint"):
        rng = np.random.default_rng(seed)
        H, W = case["H"], case["W"]
        soa = _scene(rng, case["n"], H, W, case)
        o = _optics(rng, H, W, case)
        s = dict(kind=kind, r=Renderer(H, W), soa=torch.from_numpy(soa).to(dev), optics=o)
        if kind == "adjoint":
            K = bin(case["modes"]).count("1")
            s["grad"] = _normal(torch.Generator().manual_seed(seed), (K, H, W), dev)
            s["ws"] = torch.empty(s["r"].backward_workspace_size(case["n"], K), dtype=torch.uint8,
                                  device=dev)
        return s
    if kind == "batch":
        soas, optics = _batch_scenes(case, seed)
        soa, offsets = scenes.concat(soas)
        return dict(kind=kind, r=Renderer(case["size"], case["size"]),
                    soa=torch.from_numpy(soa).to(dev), offsets=offsets, optics=optics)
    if kind == "loss":
        gen = torch.Generator().manual_seed(seed)
        shape = (case["K"], case["H"], case["W"])
        target, image = (_smooth_images(gen, shape, dev) for _ in range(2))
        fn = inverse.ImageLoss(Renderer(case["H"], case["W"]), target, 0.5,
                               spectral_weight=case["spectral"])
        fn.cutoff.fill_(2.0 * case["cut_na"] / 0.55)
        return dict(kind=kind, fn=fn, image=(0.7 * target + 0.3 * image).contiguous())
    if kind == "noise":
        gen = torch.Generator().manual_seed(seed)
        image = _smooth_images(gen, (case["S"], case["H"], case["W"]), dev)
        return dict(kind=kind, image=image, photons=case["photons"], sigma=case["sigma"],
                    seed=seed)
    if kind == "conv":
        x, w, b, dy = _conv_tensors(case, seed, dev)
        return dict(kind=kind, x=x, w=w, b=b, dy=dy, stride=case["stride"], pad=case["R"] // 2)
    w, b, x, dout = _net_tensors(case, seed, dev)
    net = cnn.WarmStartNet(dev)
    net.w, net.b = w, b
    net.refresh()
    return dict(kind=kind, net=net, x=x, dout=dout)


# ------------------------------------------------------------------ one pass
def run(state):
    kind = state["kind"]
    if kind == "render":
        return state["r"].render(state["soa"], None, state["optics"])
    if kind == "batch":
        return state["r"].batch(state["soa"], state["offsets"], state["optics"])
    if kind == "adjoint":
        r = state["r"]
        image, ws = r.render_keep(state["soa"], None, state["optics"], ws=state["ws"])
        gsoa, gopt = r.backward_kept(state["soa"], None, state["optics"], state["grad"], ws)
        return image, gsoa, gopt
    if kind == "loss":
        return state["fn"](state["image"])
    if kind == "noise":
        return noise.sensor_noise(state["image"], state["photons"], state["sigma"], state["seed"])
    if kind == "conv":
        x, w, dy, st, pad = (state[k] for k in ("x", "w", "dy", "stride", "pad"))
        y = cnn.conv2d(x, w, state["b"], st, pad, relu=True)
        dx = cnn.conv2d_backward_data(dy, w, tuple(x.shape), st, pad, x_act=x)
        dw, db = cnn.conv2d_backward_filter(dy, x, tuple(w.shape), st, pad)
        return y, dx, dw, db
    out, acts = state["net"].forward(state["x"])
    if kind == "infer":
        return out
    grads = state["net"].backward(state["dout"], acts)
    return out, [g[0] for g in grads], [g[1] for g in grads]


# ------------------------------------------------------------------ work
def _conv_work(N, H, W, C, K, R, st, pad):
    """Multiply-adds of one product and the elements of its three tensors."""
    P, Q = (H + 2 * pad - R) // st + 1, (W + 2 * pad - R) // st + 1
    return N * P * Q * K * R * R * C, N * H * W * C, K * R * R * C, N * P * Q * K, (P, Q)


def work(case):
    kind = case["kind"]
    fft = lambda H, W: 5.0 * H * W * math.log2(H * W)  # noqa: E731
    if kind in ("render", "adjoint", "batch"):
        K = bin(case["modes"]).count("1")
        H, W = (case["size"],) * 2 if kind == "batch" else (case["H"], case["W"])
        S = case.get("S", 1)
        n = case["n"] if kind != "batch" else \
            S * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"]) \
            if case["hi"] > case["lo"] else S * case["hi"]
        area = 130.0 * case["scale"] ** 2  # mean footprint in pixels
        flops = S * ((1 + K) * fft(H, W) + 30.0 * (1 + K) * H * W) + 15.0 * n * area
        bytes_ = 36.0 * n + 4.0 * S * K * H * W
        if kind == "adjoint":
            flops = 2.0 * flops + K * fft(H, W) + 40.0 * n * area
            bytes_ = 2.0 * bytes_
        return dict(bytes=bytes_, flops=flops)
    if kind == "loss":
        px = case["K"] * case["H"] * case["W"]
        return dict(bytes=px * (4.0 + 8.0 + 4.0),
                    flops=case["K"] * (2 * fft(case["H"], case["W"])) + 30.0 * px)
    if kind == "noise":
        px = case["S"] * case["H"] * case["W"]
        return dict(bytes=8.0 * px, flops=200.0 * px)
    if kind == "conv":
        m, x, w, y, _ = _conv_work(case["N"], case["H"], case["W"], case["C"], case["K"],
                                   case["R"], case["stride"], case["R"] // 2)
        return dict(bytes=2.0 * (2 * x + 2 * y + w) + 4.0 * w, flops=6.0 * m)
    flops = bytes_ = 0.0
    H, W = case["H"], case["W"]
    for i, (cin, cout, k, st, pad) in enumerate(_net_specs()):
        m, x, w, y, (H, W) = _conv_work(case["N"], H, W, cin, cout, k, st, pad)
        if i == 0:
            bytes_ += 2.0 * x
        bytes_ += 2.0 * w
        flops += 2.0 * m if kind == "infer" else (4.0 if i == 0 else 6.0) * m
        if kind == "net":
            bytes_ += 4.0 * w
    return dict(bytes=bytes_ + 4.0 * y, flops=flops)


# ------------------------------------------------------------------ float64
def _thickness(p, ex, ey, slope_dx):
    """Chord (um) of every particle at the offsets (ex, ey) from its centre."""
    c, s = torch.cos(p[2])[:, None, None], torch.sin(p[2])[:, None, None]
    a, b, T = (p[i][:, None, None] for i in (3, 4, 5))
    u, v = c * ex + s * ey, c * ey - s * ex
    d = 1.0 - (u / a) ** 2 - (v / b) ** 2
    inside = d > 0
    ell = T * torch.where(inside, torch.where(inside, d, 1.0).sqrt(), 0.0)
    wall = torch.minimum(a - u.abs(), b - v.abs())
    prism = torch.minimum((2.0 * slope_dx * wall).clamp(min=0.0), T.expand_as(wall))
    return torch.where(p[8][:, None, None] > 0.5, prism, ell)


def _compose(soa, H, W, o):
    """OPD and attenuation maps of (9, n) float64 particles."""
    opd = torch.zeros(H * W, dtype=torch.float64, device=soa.device)
    att = torch.zeros_like(opd)
    half = int(math.ceil(float(torch.hypot(soa[3], soa[4]).max()))) + 1 if soa.shape[1] else 0
    grid = torch.arange(-half, half + 1, device=soa.device)
    step = max(1, 12_000_000 // (2 * half + 1) ** 2)
    for k in range(0, soa.shape[1], step):
        p = soa[:, k:k + step]
        xs = torch.floor(p[0].detach()).long()[:, None, None] + grid[None, None, :]
        ys = torch.floor(p[1].detach()).long()[:, None, None] + grid[None, :, None]
        t = _thickness(p, xs + 0.5 - p[0][:, None, None], ys + 0.5 - p[1][:, None, None],
                       o["bevel_slope"] * o["dx"])
        on = (xs >= 0) & (xs < W) & (ys >= 0) & (ys < H) & (t.detach() > 0)
        at = (ys * W + xs)[on]
        who = torch.arange(p.shape[1], device=soa.device)[:, None, None].expand_as(on)[on]
        t = t[on]
        opd = opd.index_add(0, at, t * p[6][who])
        att = att.index_add(0, at, t * p[7][who])
    return opd.view(H, W), att.view(H, W)


def _images(soa, o, scalars):
    """(K, H, W) float64 images; scalars are (defocus, shear_px, shear_angle,
    bias) as tensors."""
    H, W = o["H"], o["W"]
    dev = soa.device
    opd, att = _compose(soa, H, W, o)
    phase = 2.0 * math.pi * opd / o["lambda_um"]
    spec = torch.fft.fft2(torch.polar(torch.exp(-att), phase))
    del opd, att, phase
    fx = torch.fft.fftfreq(W, dtype=torch.float64, device=dev)[None, :] / o["dx"]
    fy = torch.fft.fftfreq(H, dtype=torch.float64, device=dev)[:, None] / o["dx"]
    dz, shear, angle, bias = scalars
    k0 = 2.0 * math.pi * o["n_medium"] / o["lambda_um"]
    cut = o["NA"] / o["lambda_um"]
    out = []
    for mode in (BF, OBLIQUE, DIC):
        if not o["modes"] & mode:
            continue
        ox = oy = 0.0
        if mode == OBLIQUE:
            ox = o["oblique_frac"] * cut * math.cos(o["oblique_angle"])
            oy = o["oblique_frac"] * cut * math.sin(o["oblique_angle"])
        q2 = (fx + ox) ** 2 + (fy + oy) ** 2
        circ = q2 <= cut * cut
        q2 = torch.where(circ, q2, 0.0) * (4.0 * math.pi ** 2)
        chi = -dz * q2 / (torch.sqrt(k0 * k0 - q2) + k0)
        h = torch.polar(circ.double(), chi)
        if mode == DIC:
            half = 0.5 * shear * o["dx"] * 2.0 * math.pi
            a = half * (fx * torch.cos(angle) + fy * torch.sin(angle)) + bias
            h = h * (2j * torch.sin(a))
        e = torch.fft.ifft2(spec * h)
        out.append(e.real ** 2 + e.imag ** 2)
    return torch.stack(out)


def _scalars(o, dev, grad=False):
    return [torch.tensor(float(o[k]), dtype=torch.float64, device=dev, requires_grad=grad)
            for k in OPTICS_GRADS]


def _exact_loss(s, case):
    image, target = s["image"].double(), s["fn"].target.double()
    K, H, W = image.shape
    A, B = torch.fft.fft2(image), torch.fft.fft2(target)
    fx = torch.fft.fftfreq(W, dtype=torch.float64, device=image.device)[None, :] / 0.5
    fy = torch.fft.fftfreq(H, dtype=torch.float64, device=image.device)[:, None] / 0.5
    low = fx * fx + fy * fy <= float(s["fn"].cutoff) ** 2
    D = torch.where(low, A - B, 0.0)
    scale = 1.0 / (K * H * W)
    misfit = (D.abs() ** 2).sum() * scale / (H * W)
    grad = 2.0 * scale / (H * W) * D
    eps = 1e-4 * B.abs().amax(dim=(1, 2), keepdim=True)
    spectral = torch.zeros((), dtype=torch.float64, device=image.device)
    if case["spectral"]:
        ma = A.abs()
        d = torch.log(ma + eps) - torch.log(B.abs() + eps)
        spectral = (d * d).mean()
        safe = torch.where(ma > 0, ma, 1.0)
        grad = grad + torch.where(ma > 0, 2.0 * case["spectral"] / (K * H * W) * d
                                  / (safe * (safe + eps)), 0.0) * A
    return torch.stack([misfit, spectral]), (torch.fft.ifft2(grad) * (H * W)).real


_MASK = 0xFFFFFFFF


def _mulhilo(a, m):
    """High and low words of the 32-bit product of a tensor and a constant."""
    low, high = (a & 0xFFFF) * m, (a >> 16) * m
    mid = high + (low >> 16)
    return mid >> 16, ((mid & 0xFFFF) << 16) | (low & 0xFFFF)


def _uniforms(index, rnd, seed):
    """Four uniforms in (0, 1) of Philox4x32-10 (Salmon et al., SC 2011) with
    the counter (element, round, tag) and the seed as the key."""
    c = [index & _MASK, index >> 32, torch.full_like(index, rnd),
         torch.full_like(index, 0x6E6F6973)]
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK
    for _ in range(10):
        h0, l0 = _mulhilo(c[0], 0xD2511F53)
        h1, l1 = _mulhilo(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return [(v.double() + 0.5) / 4294967296.0 for v in c]


def _poisson(lam, index, u, seed):
    k = torch.zeros_like(lam)
    few = (lam > 0) & (lam < 10.0)
    if few.any():  # inversion by sequential search
        l, x = lam[few], u[2][few]
        p = torch.exp(-l)
        f, n = p.clone(), torch.zeros_like(l)
        while True:
            more = x > f
            if not more.any() or float(n.max()) >= 200:
                break
            n = torch.where(more, n + 1, n)
            p = torch.where(more, p * l / n.clamp(min=1.0), p)
            f = torch.where(more, f + p, f)
        k[few] = n
    at = torch.nonzero(lam >= 10.0).view(-1)
    for rnd in range(64):  # Hormann's transformed rejection (PTRS, 1993)
        if not at.numel():
            break
        us = u if rnd == 0 else None
        if rnd == 0:
            us = [v[at] for v in u]
        else:
            us = _uniforms(index[at], rnd, seed)
        for pair in ((1,) if rnd == 0 else (0, 1)):
            l = lam[at]
            b = 0.931 + 2.53 * torch.sqrt(l)
            a = -0.059 + 0.02483 * b
            U, V = us[2 * pair] - 0.5, us[2 * pair + 1]
            w = 0.5 - U.abs()
            n = torch.floor((2.0 * a / w + b) * U + l + 0.43)
            quick = (w >= 0.07) & (V <= 0.9277 - 3.6224 / (b - 2.0))
            no = (n < 0) | ((w < 0.013) & (V > w))
            inv = 1.1239 + 1.1328 / (b - 3.4)
            slow = torch.log(V * inv / (a / (w * w) + b)) <= \
                -l + n * torch.log(l) - torch.lgamma(n.clamp(min=0.0) + 1.0)
            yes = quick | (~no & slow)
            k[at[yes]] = n[yes]
            at, us = at[~yes], [v[~yes] for v in us]
    return k


def _exact_noise(s):
    flat = s["image"].reshape(-1)
    g, sigma, seed = s["photons"], s["sigma"], s["seed"]
    out = torch.empty(flat.shape, dtype=torch.float64, device=flat.device)
    for i in range(0, flat.numel(), 1 << 21):
        index = torch.arange(i, min(i + (1 << 21), flat.numel()), device=flat.device)
        u = _uniforms(index, 0, seed)
        lam = g * flat[index].double().clamp(min=0.0)
        z = torch.sqrt(-2.0 * torch.log(u[0])) * torch.cos(2.0 * math.pi * u[1])
        out[index] = (_poisson(lam, index, u, seed) + sigma * z) / g
    return out.view(s["image"].shape)


def _conv64(x, w, st, pad):
    """NHWC convolution in float64 as one matrix product per filter tap."""
    N, H, W, C = x.shape
    K, R, S, _ = w.shape
    P, Q = (H + 2 * pad - R) // st + 1, (W + 2 * pad - S) // st + 1
    xp = F.pad(x, (0, 0, pad, pad, pad, pad))
    y = torch.zeros((N * P * Q, K), dtype=torch.float64, device=x.device)
    for r in range(R):
        for s in range(S):
            v = xp[:, r:r + (P - 1) * st + 1:st, s:s + (Q - 1) * st + 1:st]
            y.addmm_(v.reshape(-1, C), w[:, r, s].t())
    return y.view(N, P, Q, K)


def _conv64_grads(x, w, dy, st, pad, need_dx=True):
    N, H, W, C = x.shape
    K, R, S, _ = w.shape
    P, Q = dy.shape[1:3]
    xp = F.pad(x, (0, 0, pad, pad, pad, pad))
    dxp = torch.zeros_like(xp) if need_dx else None
    dw = torch.empty(w.shape, dtype=torch.float64, device=x.device)
    d = dy.reshape(-1, K)
    for r in range(R):
        for s in range(S):
            at = (slice(None), slice(r, r + (P - 1) * st + 1, st),
                  slice(s, s + (Q - 1) * st + 1, st))
            dw[:, r, s] = d.t() @ xp[at].reshape(-1, C)
            if need_dx:
                dxp[at] += (d @ w[:, r, s]).view(N, P, Q, C)
    dx = dxp[:, pad:pad + H, pad:pad + W] if need_dx else None
    return dx, dw, d.sum(0)


def _bf16(t):
    return t.to(torch.bfloat16).double()


def _exact_net(case, seed, dev):
    """The network in float64, its activations and their gradients stored in
    bfloat16 between the layers as everywhere in the framework."""
    w, b, x, dout = _net_tensors(case, seed, dev)
    w = [_bf16(v) for v in w]
    specs = _net_specs()
    acts = [x.double()]
    for i, (_, _, _, st, pad) in enumerate(specs):
        y = _conv64(acts[-1], w[i], st, pad) + b[i].double()
        if i < len(specs) - 1:
            acts.append(_bf16(y.clamp(min=0.0)))
    if case["kind"] == "infer":
        return y
    dws, dbs, dy = [], [], _bf16(dout)
    for i in reversed(range(len(specs))):
        _, _, _, st, pad = specs[i]
        dx, dw, db = _conv64_grads(acts[i], w[i], dy, st, pad, need_dx=i > 0)
        dws.insert(0, dw)
        dbs.insert(0, db)
        if i > 0:
            dy = _bf16(dx * (acts[i] > 0))
    return y, dws, dbs


def exact(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind in ("net", "infer"):
        return _exact_net(case, seed, dev)
    if kind == "batch":
        soas, optics = _batch_scenes(case, seed)
        return torch.stack([_images(torch.from_numpy(p).to(dev).double(), o, _scalars(o, dev))
                            for p, o in zip(soas, optics)])
    s = prepare(case, seed)
    if kind == "render":
        return _images(s["soa"].double(), s["optics"], _scalars(s["optics"], dev))
    if kind == "adjoint":
        soa = s["soa"].double().requires_grad_(True)
        scalars = _scalars(s["optics"], dev, grad=True)
        image = _images(soa, s["optics"], scalars)
        image.backward(s["grad"].double())
        gopt = torch.stack([torch.zeros_like(v) if v.grad is None else v.grad for v in scalars])
        return image.detach(), soa.grad, gopt
    if kind == "loss":
        return _exact_loss(s, case)
    if kind == "noise":
        return _exact_noise(s)
    x, w, b, dy = (s[k].double() for k in ("x", "w", "b", "dy"))
    y = (_conv64(x, w, s["stride"], s["pad"]) + b).clamp(min=0.0)
    dx, dw, db = _conv64_grads(x, w, dy, s["stride"], s["pad"])
    return y, dx * (x > 0), dw, db
