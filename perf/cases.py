"""What the performance of this library is measured on: the calls a program makes, from one small frame to a
batch of 32 views of three million Gaussians, through the package's public entry points.

A case's ``kind`` names the call:

* ``view``    forward only (a viewer, the render server's inner call): ``Renderer.render``;
* ``step``    render + path-replay backward: ``Renderer.render`` and ``Renderer.backward``;
* ``autograd`` the same through the differentiable ``render`` function;
* ``views``   several cameras of one scene in one call (``Renderer.render_batch``), with or without backward;
* ``loss``    the training image loss and its gradient (``train.l1_ssim``);
* ``adam``    one optimizer step over the five parameter arrays (``train.Adam.step``);
* ``train``   a whole training step (``train.Trainer.step``);
* ``densify`` split / prune of a model with its optimizer state (``train.densify``).
"""
import math

import numpy as np
import torch

from paper_2603_02887_gb300 import render as R
from paper_2603_02887_gb300 import synth
from paper_2603_02887_gb300 import train as T

KEYS = R.PARAM_KEYS
DEV = "cuda"


def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, scene="clustered", n=0, degree=3, width=0, height=0, model="sup", tile_w=16,
             tile_h=16, chunk=0, schedule="tiles", graphs=False, asynchronous=False, views=1, backward=True)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest frame of the tests and the benchmark: launches and host calls are all there is
        _case("tiny_exp", "step", scene="tiny", n=1000, degree=0, width=128, height=128, model="exp"),
        # a small scene through autograd, with one of the other transmittance models, ragged tiles
        _case("autograd_blend_20k", "autograd", n=20000, width=325, height=243, model="blend"),
        # a viewer at full resolution with the default options
        _case("view_sup_500k", "view", n=500_000, width=1920, height=1080, model="sup", backward=False),
        # the benchmark's step in the options it tunes for the exponential model: graphs, asynchronous frames
        _case("step_exp_500k", "step", n=500_000, width=1920, height=1080, model="exp", tile_w=8, tile_h=8, chunk=32,
              schedule="persistent", graphs=True, asynchronous=True),
        # the same frame with the sub-linear model, as a program that calls the two functions and nothing else
        _case("step_sub_500k", "step", n=500_000, width=1920, height=1080, model="sub", chunk=128,
              schedule="persistent"),
        # the differentiation configuration: one million Gaussians, a width that fills no tile row
        _case("step_lin_1m", "step", n=1_000_000, width=1297, height=840, model="lin"),
        # what the render server does with requests for one scene: several views of uneven sizes, forward only
        _case("views8_sup_1m", "views", n=1_000_000, views=8, model="sup", schedule="persistent", backward=False),
        # the batched configuration: three million Gaussians, 32 views of uneven sizes, with gradients
        _case("views32_exp_3m", "views", n=3_000_000, views=32, model="exp", tile_w=8, tile_h=8),
        # the image loss of a training step at full resolution
        _case("loss_1080p", "loss", width=1920, height=1080),
        # the optimizer step of a million Gaussians
        _case("adam_1m", "adam", n=1_000_000),
        # one step of the training driver at the benchmark's training size
        _case("train_sup_50k", "train", n=50_000, width=640, height=360, model="sup", views=8),
        # split / prune of a model on its way to the primitive cap that the training driver defaults to
        _case("densify_100k", "densify", n=100_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo=96, hi=1920):
    w = _log(rng, lo, hi)
    return w, max(16, int(w * rng.uniform(0.5, 1.0)))


def draw(rng):
    kind = rng.choice(["view", "view", "step", "step", "step", "autograd", "views", "views", "loss", "adam", "train",
                       "densify"])
    if kind == "adam":
        return _unnamed(kind, n=_log(rng, 1000, 3_000_000), degree=rng.randint(0, 3))
    if kind == "densify":
        return _unnamed(kind, n=_log(rng, 1000, 500_000), degree=rng.randint(0, 3))
    w, h = _size(rng)
    if kind == "loss":
        return _unnamed(kind, width=w, height=h)
    model = rng.choice(["exp", "sub", "lin", "sup", "exp", "sub", "lin", "sup", "blend", "vicini"])
    if kind == "train":
        return _unnamed(kind, n=_log(rng, 5000, 200_000), width=w // 2, height=h // 2, model=model,
                        views=rng.randint(2, 8))
    tile_w, tile_h = rng.choice([(8, 8), (16, 16), (16, 16), (16, 32)])
    opts = dict(model=model, tile_w=tile_w, tile_h=tile_h, schedule=rng.choice(["tiles", "persistent"]),
                degree=rng.randint(0, 3))
    if kind == "views":
        return _unnamed(kind, n=_log(rng, 10_000, 1_000_000), views=rng.randint(2, 12),
                        backward=rng.random() < 0.5, **opts)
    if kind == "autograd":
        return _unnamed(kind, n=_log(rng, 2000, 300_000), width=w, height=h, **opts)
    return _unnamed(kind, n=_log(rng, 1000, 2_000_000), width=w, height=h, backward=kind == "step",
                    graphs=rng.random() < 0.4, asynchronous=rng.random() < 0.4, **opts)


def _unnamed(kind, **kw):
    c = _case("", kind, **kw)
    del c["name"]
    return c


# ---- inputs --------------------------------------------------------------------------------------------


def _cameras(case):
    if case["kind"] == "views":
        return synth.orbit_cameras(case["views"], radius=12.0, seed=2)
    if case["kind"] == "train":
        return synth.orbit_cameras(case["views"], radius=12.0, seed=2,
                                   resolutions=((case["width"], case["height"]),))
    if case["scene"] == "tiny":
        return [synth.tiny_camera()]
    return [synth.outside_camera(case["width"], case["height"])]


def _scene(case, seed):
    """The package's synthetic scenes (synth.py), drawn on the GPU: the same distributions."""
    n, degree = case["n"], case["degree"]
    if case["scene"] == "tiny":
        return {k: torch.from_numpy(v).to(DEV) for k, v in synth.tiny_scene(seed, n).items()}
    g = torch.Generator(device=DEV).manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(*shape, generator=g, device=DEV)

    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV)

    clusters = 64
    centres = uniform(-5.0, 5.0, clusters, 3)
    axes = torch.linalg.qr(normal(clusters, 3, 3).cpu())[0].to(DEV)
    lam = torch.exp(uniform(math.log(0.05), math.log(2.0), clusters, 3))
    which = torch.randint(0, clusters, (n,), generator=g, device=DEV)
    local = normal(n, 3) * torch.sqrt(lam[which])
    means = centres[which] + (axes[which] * local[:, None, :]).sum(-1)
    quats = normal(n, 4)
    sh = normal(n, (degree + 1) ** 2, 3) * 0.1
    sh[:, 0, :] = (torch.rand(n, 3, generator=g, device=DEV) - 0.5) * (2.0 * math.sqrt(math.pi))
    return dict(means=means.contiguous(), log_scales=-4.0 + 0.7 * normal(n, 3),
                quats=quats / quats.norm(dim=1, keepdim=True), opacity_logits=0.5 + 1.5 * normal(n), sh=sh.contiguous())


def _upstream(pixels, seed):
    """The upstream gradient of an L1 loss: +-1."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
    return torch.where(torch.rand(pixels, 3, generator=g, device=DEV) < 0.5, -1.0, 1.0)


def _options(case):
    return R.default_options(tile_w=case["tile_w"], tile_h=case["tile_h"], chunk=case["chunk"],
                             schedule=case["schedule"])


def _images(case, seed):
    """A rendered-looking image (smooth colours with some texture) and a target near it."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    h, w = case["height"], case["width"]
    coarse = torch.rand(1, 3, max(2, h // 24), max(2, w // 24), generator=g, device=DEV)
    smooth = torch.nn.functional.interpolate(coarse, size=(h, w), mode="bilinear", align_corners=False)[0]
    texture = 0.05 * torch.randn(3, h, w, generator=g, device=DEV)
    image = (smooth + texture).clamp(0, 1).permute(1, 2, 0).contiguous()
    target = (image + 0.03 * torch.randn(h, w, 3, generator=g, device=DEV)).clamp(0, 1)
    return image, target


def _random_like(params, seed, scale, positive=False):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    out = {}
    for k in KEYS:
        x = torch.randn(params[k].shape, generator=g, device=DEV) * scale
        out[k] = x * x / scale if positive else x
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "loss":
        image, target = _images(case, seed)
        return dict(case=case, renderer=R.Renderer(DEV), image=image, target=target)
    params = _scene(case, seed)
    s = dict(case=case, params=params, renderer=R.Renderer(DEV))
    if kind == "adam":
        s["grads"] = {"d_" + k: v for k, v in _random_like(params, seed + 2, 1e-3).items()}
        s["adam"] = T.Adam(params)
        s["adam"].m.update(_random_like(params, seed + 3, 1e-3))
        s["adam"].v.update(_random_like(params, seed + 4, 1e-6, positive=True))
        s["adam"].t = 100
        return s
    if kind == "densify":
        s["adam"] = T.Adam(params)
        s["adam"].m.update(_random_like(params, seed + 3, 1e-3))
        s["adam"].v.update(_random_like(params, seed + 4, 1e-6, positive=True))
        # a tenth of the Gaussians below the opacity limit, a fifth of the others above the gradient threshold
        n = case["n"]
        g = torch.Generator(device=DEV).manual_seed(int(seed) + 5)
        order = torch.randperm(n, generator=g, device=DEV)
        prune, split = order[:n // 10], order[n // 10:n // 10 + n // 5]
        params["opacity_logits"].clamp_(min=-4.5)
        params["opacity_logits"][prune] = -6.0
        norm = 2e-4 * (0.9 * torch.rand(n, generator=g, device=DEV))
        norm[split] = 2e-4 * (1.1 + torch.rand(split.shape[0], generator=g, device=DEV))
        s["count"] = torch.randint(1, 100, (n,), generator=g, device=DEV).float()
        s["accum"] = s["count"] * norm
        return s
    cams = _cameras(case)
    pixels = sum(c["width"] * c["height"] for c in cams)
    s["cams"], s["options"] = cams, _options(case)
    if kind == "train":
        targets = T.render_targets(s["renderer"], params, cams, case["model"], factors=(1,))
        g = torch.Generator(device=DEV).manual_seed(int(seed) + 6)
        start = {k: v + 0.05 * torch.randn(v.shape, generator=g, device=DEV) for k, v in params.items()}
        s["trainer"] = T.Trainer(start, cams, targets, case["model"], iters=30000, densify_until=0,
                                 coarse_to_fine=((0, 1),), options=s["options"], renderer=s["renderer"])
        return s
    if case["backward"]:
        s["dl"] = _upstream(pixels, seed)
        if kind != "views":
            s["dl"] = s["dl"].view(cams[0]["height"], cams[0]["width"], 3)
    if kind == "autograd":
        for p in params.values():
            p.requires_grad_(True)
        return s
    r = s["renderer"]
    s["frame"] = r.frame()
    s["image"] = torch.empty(pixels, 3, device=DEV)
    s["overdraw"] = torch.empty(pixels, dtype=torch.int32, device=DEV)
    if kind != "views":
        s["image"] = s["image"].view(cams[0]["height"], cams[0]["width"], 3)
        s["overdraw"] = s["overdraw"].view(cams[0]["height"], cams[0]["width"])
    if case["backward"]:
        s["grads"] = {"d_" + k: torch.empty_like(v) for k, v in params.items()}
    r.set_graphs(case["graphs"])
    if case["asynchronous"]:  # the first render of an asynchronous frame sets its capacity
        r.render(params, cams[0], case["model"], s["options"], frame=s["frame"], image=s["image"],
                 overdraw=s["overdraw"])
        s["frame"].set_async(True)
    return s


def run(s):
    case = s["case"]
    kind, r = case["kind"], s["renderer"]
    if kind == "loss":
        return {"dl_dimage": T.l1_ssim(r, s["image"], s["target"], read_loss=False)[1]}
    if kind == "adam":
        s["adam"].step(r, s["params"], s["grads"])
        return {"params": s["params"], "m": s["adam"].m, "v": s["adam"].v}
    if kind == "densify":
        adam = T.Adam.__new__(T.Adam)
        adam.m, adam.v = s["adam"].m, s["adam"].v
        new = T.densify(r, s["params"], adam, s["accum"], s["count"], grad_threshold=2e-4,
                        max_gaussians=2 * case["n"])
        return {"params": new, "m": adam.m, "v": adam.v}
    if kind == "train":
        t = s["trainer"]
        t.step()
        return {"params": t.params, "m": t.adam.m, "v": t.adam.v, "accum": t.accum}
    if kind == "autograd":
        image, overdraw = R.render(s["params"], s["cams"][0], case["model"], s["options"], renderer=r)
        grads = torch.autograd.grad(image, [s["params"][k] for k in KEYS], s["dl"])
        return {"image": image, "overdraw": overdraw, "grads": {"d_" + k: g for k, g in zip(KEYS, grads)}}
    if kind == "views":
        r.render_batch(s["params"], s["cams"], case["model"], s["options"], frame=s["frame"], images=s["image"],
                       overdraw=s["overdraw"])
    else:
        r.render(s["params"], s["cams"][0], case["model"], s["options"], frame=s["frame"], image=s["image"],
                 overdraw=s["overdraw"])
    out = {"image": s["image"], "overdraw": s["overdraw"]}
    if case["backward"]:
        out["grads"] = r.backward(s["frame"], s["params"], s["dl"], out=s["grads"])
    return out


# ---- the work a pass cannot do without -----------------------------------------------------------------


def work(case):
    kind, n = case["kind"], case["n"]
    coef = 3 * (case["degree"] + 1) ** 2
    row = 4 * (11 + coef)  # bytes of one Gaussian's parameters
    if kind == "loss":
        px = case["width"] * case["height"]  # two images in, one gradient out; 8 separable 11-tap windows
        return {"bytes": 36.0 * px, "flops": 3.0 * px * (8 * 22 * 2 + 60)}
    if kind == "adam":  # parameters and both moments read and written, gradients read
        return {"bytes": 7.0 * row * n, "flops": 15.0 * (row / 4) * n}
    if kind == "densify":  # parameters and both moments read; nine tenths of the Gaussians and a fifth more written
        return {"bytes": (3.0 + 3.0 * 1.1) * row * n + 8.0 * n, "flops": 20.0 * n}
    cams = _cameras(case)
    if kind == "train":
        cams = cams[:1]
    px = sum(c["width"] * c["height"] for c in cams)
    # splats composited per pixel: about 34 for 500k Gaussians and the exponential model, at most about 8 once
    # rays saturate (the quadratic models), in proportion to the Gaussians below that
    cover = 34.0 * n / 500_000 if case["scene"] != "tiny" else 12.0
    per_px = min(cover, 60.0 if case["model"] in ("exp", "vicini", "blend") else 8.0)
    bytes_, flops = row * n + 16.0 * px, 250.0 * n * len(cams) + 22.0 * per_px * px
    if case["backward"]:
        bytes_ += row * n + 12.0 * px
        flops += 700.0 * n * len(cams) + 55.0 * per_px * px
    if kind == "train":
        loss = work(dict(case, kind="loss"))
        opt = work(dict(case, kind="adam"))
        bytes_ += loss["bytes"] + opt["bytes"]
        flops += loss["flops"] + opt["flops"]
    return {"bytes": float(bytes_), "flops": float(flops)}


# ---- the same in 64 bits, in plain torch ----------------------------------------------------------------


def _f32(x):
    return float(np.float32(x))


MODELS64 = {"exp": (0, 0.0), "sub": (1, -0.5), "lin": (1, 0.0), "sup": (1, 0.5), "blend": (2, 0.5), "vicini": (3, 0.5)}
RATES64 = (1.6e-3, 5e-3, 1e-3, 5e-2, 2.5e-3)
ALPHA_MIN, ALPHA_MAX, T_EPS, DILATION, NEAR = _f32(1 / 255), _f32(0.99), _f32(1e-4), _f32(0.3), _f32(0.2)


def _sh_basis(degree, d):
    x, y, z = d.unbind(-1)
    pi = math.pi
    b = [torch.full_like(x, math.sqrt(1 / (4 * pi)))]
    if degree > 0:
        c = math.sqrt(3 / (4 * pi))
        b += [-c * y, c * z, -c * x]
    if degree > 1:
        c = math.sqrt(15 / (4 * pi))
        b += [c * x * y, -c * y * z, math.sqrt(5 / (16 * pi)) * (2 * z * z - x * x - y * y), -c * x * z,
              0.5 * c * (x * x - y * y)]
    if degree > 2:
        a, e, f = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi)), math.sqrt(21 / (32 * pi))
        b += [-a * y * (3 * x * x - y * y), e * x * y * z, -f * y * (4 * z * z - x * x - y * y),
              math.sqrt(7 / (16 * pi)) * z * (2 * z * z - 3 * x * x - 3 * y * y), -f * x * (4 * z * z - x * x - y * y),
              0.5 * e * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(b, -1)


def _project64(p, cam, degree):
    """Screen mean, conic, opacity and colour of every Gaussian, and the FP32 depth that orders them."""
    vm = torch.from_numpy(np.asarray(cam["viewmat"], np.float32).reshape(3, 4).astype(np.float64)).to(DEV)
    rot, t = vm[:, :3], vm[:, 3]
    fx, fy, cx, cy = (_f32(cam[k]) for k in ("fx", "fy", "cx", "cy"))
    v = p["means"] @ rot.T + t
    x, y, z = v.unbind(-1)
    q = p["quats"] / p["quats"].norm(dim=1, keepdim=True)
    w, a, b, c = q.unbind(-1)
    rq = torch.stack([1 - 2 * (b * b + c * c), 2 * (a * b - w * c), 2 * (a * c + w * b), 2 * (a * b + w * c),
                      1 - 2 * (a * a + c * c), 2 * (b * c - w * a), 2 * (a * c - w * b), 2 * (b * c + w * a),
                      1 - 2 * (a * a + b * b)], -1).view(-1, 3, 3)
    m = rq * torch.exp(p["log_scales"])[:, None, :]
    zero = torch.zeros_like(z)
    jac = torch.stack([fx / z, zero, -fx * x / z ** 2, zero, fy / z, -fy * y / z ** 2], -1).view(-1, 2, 3)
    u = jac @ (rot @ m)
    cov = u @ u.transpose(1, 2)
    s00, s01, s11 = cov[:, 0, 0] + DILATION, cov[:, 0, 1], cov[:, 1, 1] + DILATION
    det = s00 * s11 - s01 * s01
    dirs = p["means"] + rot.T @ t
    dirs = dirs / dirs.norm(dim=1, keepdim=True)
    rgb = (0.5 + torch.einsum("nk,nkc->nc", _sh_basis(degree, dirs), p["sh"])).clamp(min=0)
    rec = torch.cat([torch.stack([fx * x / z + cx, fy * y / z + cy, s11 / det, -s01 / det, s00 / det,
                                  torch.sigmoid(p["opacity_logits"])], -1), rgb], 1)
    with torch.no_grad():
        z32 = t[2].float()
        for k in range(3):
            z32 = (rot[2, k] * p["means"][:, k] + z32.double()).float()
    return rec, z32


def _alpha64(rec, px, py):
    dx, dy = px - rec[:, None, 0], py - rec[:, None, 1]
    power = -0.5 * (rec[:, None, 2] * dx * dx + rec[:, None, 4] * dy * dy) - rec[:, None, 3] * dx * dy
    return rec[:, None, 5] * torch.exp(power)


def _weights64(raw, model):
    """Contribution of each splat (rows, front to back) at each pixel (columns)."""
    kind, par = MODELS64[model]
    a = torch.where(raw >= ALPHA_MIN, raw.clamp(max=ALPHA_MAX), torch.zeros_like(raw))
    through = torch.exp(torch.cumsum(torch.log1p(-a), 0))
    before = torch.cat([torch.ones_like(through[:1]), through[:-1]])

    def saturate(pt):
        total = torch.cumsum(pt, 0)
        prev = total - pt
        over = (total >= 1.0) & (raw >= ALPHA_MIN)
        earlier = torch.cumsum(over.to(torch.int32), 0) - over.to(torch.int32)
        return torch.where(earlier > 0, torch.zeros_like(pt), torch.where(over, 1.0 - prev, pt))

    def exponential():
        return torch.where(through >= T_EPS, a * before, torch.zeros_like(a))

    if kind == 0:
        return exponential()
    if kind == 1:
        tau = torch.cumsum(a, 0) - a
        return saturate((a * (1.0 + _f32(par) * tau)).clamp(min=0))
    g = _f32(par)
    if kind == 2:
        return saturate(a * (1.0 - g + g * before))
    return (1.0 - g) * saturate(a) + g * exponential()


def _render64(case, seed):
    cam = _cameras(case)[0]
    W, H = cam["width"], cam["height"]
    p = {k: v.detach().double().requires_grad_(True) for k, v in _scene(case, seed).items()}
    rec_graph, z32 = _project64(p, cam, case["degree"])
    rec = rec_graph.detach().requires_grad_(True)
    near = z32 > NEAR
    order = torch.sort(torch.where(near, z32, torch.full_like(z32, 3e38)), stable=True)[1]
    order = order[near[order]]
    image = torch.zeros(H, W, 3, dtype=torch.float64, device=DEV)
    dl = _upstream(W * H, seed).view(H, W, 3).double() if case["backward"] else None
    step = 32
    for y0 in range(0, H, step):
        for x0 in range(0, W, step):
            ys = torch.arange(y0, min(H, y0 + step), device=DEV).double() + 0.5
            xs = torch.arange(x0, min(W, x0 + step), device=DEV).double() + 0.5
            py, px = (g.reshape(1, -1) for g in torch.meshgrid(ys, xs, indexing="ij"))
            with torch.no_grad():
                hit = (_alpha64(rec[order], px, py) >= ALPHA_MIN).any(1)
            mine = rec[order[hit]]
            if mine.shape[0] == 0:
                continue
            color = _weights64(_alpha64(mine, px, py), case["model"]).T @ mine[:, 6:9]
            block = (slice(y0, y0 + len(ys)), slice(x0, x0 + len(xs)))
            image[block] = color.detach().view(len(ys), len(xs), 3)
            if dl is not None:
                color.backward(dl[block].reshape(-1, 3))
    out = {"image": image, "overdraw": None}
    if dl is not None:
        rec_graph.backward(rec.grad if rec.grad is not None else torch.zeros_like(rec))
        out["grads"] = {"d_" + k: p[k].grad for k in KEYS}
    return out


def _loss64(case, seed):
    image, target = _images(case, seed)
    x = image.double().permute(2, 0, 1).requires_grad_(True)
    y = target.double().permute(2, 0, 1)
    taps = torch.exp(-((torch.arange(11, device=DEV).double() - 5) ** 2) / (2 * 1.5 ** 2))
    taps = taps / taps.sum()

    def blur(m):
        h, w = m.shape[1:]
        pad = torch.nn.functional.pad(m, (5, 5))
        m = sum(taps[i] * pad[:, :, i:i + w] for i in range(11))
        pad = torch.nn.functional.pad(m, (0, 0, 5, 5))
        return sum(taps[i] * pad[:, i:i + h, :] for i in range(11))

    mx, my = blur(x), blur(y)
    sxx, syy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = ((2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sxx + syy + c2))).mean()
    loss = 0.8 * (x - y).abs().mean() + 0.2 * (1 - ssim)
    return {"dl_dimage": torch.autograd.grad(loss, x)[0].permute(1, 2, 0).contiguous()}


def _adam64(case, seed):
    params = _scene(case, seed)
    grads = _random_like(params, seed + 2, 1e-3)
    m, v = _random_like(params, seed + 3, 1e-3), _random_like(params, seed + 4, 1e-6, positive=True)
    b1, b2, eps, t = _f32(0.9), _f32(0.999), _f32(1e-15), 101
    out = {"params": {}, "m": {}, "v": {}}
    for k, lr in zip(KEYS, RATES64):
        lr, g = _f32(lr), grads[k].double()
        out["m"][k] = b1 * m[k].double() + (1 - b1) * g
        out["v"][k] = b2 * v[k].double() + (1 - b2) * g * g
        step = lr * (out["m"][k] / (1 - b1 ** t)) / (torch.sqrt(out["v"][k] / (1 - b2 ** t)) + eps)
        out["params"][k] = params[k].double() - step.clamp(-lr, lr)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "loss":
        return _loss64(case, seed)
    if kind == "adam":
        return _adam64(case, seed)
    # every Gaussian against every pixel: only for the small frames
    if kind in ("view", "step", "autograd") and case["n"] * case["width"] * case["height"] <= 4e9:
        return _render64(case, seed)
    return None
