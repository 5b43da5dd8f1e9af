"""The work that the measurements of this repository time: whole calls of its public entry points.

A case is a dict of plain values. ``prepare`` makes what a user's program holds before the call
(parameters, views, targets, and the rasterizer, frame or optimiser it keeps), on the GPU, from a
seed; ``run`` is one pass through the entry points; ``exact`` is the same result in 64 bits by plain
torch. Kinds of case:

  view      render(...) without gradients: novel views, a viewer, an evaluation run
  autograd  render(...) and the backward pass through torch autograd, with a given dL/dimage
  graph     GraphedFrame.replay(): forward, L1 loss and backward of all views as one CUDA graph
  grouped   GroupedFrame.step(): the same in groups of views that share one pair buffer
  loss      the L1 + D-SSIM loss and its gradient (l1_dssim)
  adam      one GaussianAdam step over the five parameter tensors
  densify   densify.select and densify.apply on accumulated statistics
"""
import math

import torch

from paper_2410_20686_gb300 import densify as D
from paper_2410_20686_gb300.graph import GraphedFrame, GroupedFrame
from paper_2410_20686_gb300.loss import l1_dssim
from paper_2410_20686_gb300.optim import GaussianAdam
from paper_2410_20686_gb300.rasterizer import Rasterizer, RenderSettings, render
from paper_2410_20686_gb300.scenes import View, cubemap_views, yaw_view

NAMES = ("means", "scales", "quats", "opacity", "sh")
DILATION, NEAR, FAR = 0.3, 0.2, 1e4  # the rasterizer's default settings


def _case(name, kind, n, width, height, *, scene="room", sh=3, views=1, mixed=False, cube=False, raw=False, bg=0.0,
          group=0, log_scale=-4.0):
    return dict(name=name, kind=kind, n=n, width=width, height=height, scene=scene, sh=sh, views=views, mixed=mixed,
                cube=cube, raw=raw, bg=bg, group=group, log_scale=log_scale)


def listed():
    return [
        # the smallest scene, seen once: a unit test, a first look at an initial point cloud
        _case("view_1k_256x128", "view", 1000, 256, 128, scene="shell", sh=0, log_scale=-3.0),
        # an early step of a small fit: every pass is launches and latency
        _case("autograd_5k_512x256", "autograd", 5000, 512, 256, scene="shell", sh=1, log_scale=-3.0),
        # one frame of a viewer on a small room
        _case("view_100k_1024x512", "view", 100_000, 1024, 512, scene="smallroom", log_scale=-3.0),
        # a training step on raw variables at sizes that nothing divides: odd counts, a last tile row of
        # one pixel row, SH degree 2 (27 floats a row), a background colour
        _case("autograd_77777_1200x593", "autograd", 77_777, 1200, 593, scene="room", sh=2, raw=True, bg=0.25,
              log_scale=-3.5),
        # evaluation of a trained model at full size
        _case("view_1m_2048x1024", "view", 1_000_000, 2048, 1024, scene="polar"),
        # the training step at full size: one view a step
        _case("graph_1m_2048x1024", "graph", 1_000_000, 2048, 1024, scene="polar"),
        # a batch of 16 views of three sizes in one frame
        _case("graph_500k_16views", "graph", 500_000, 2048, 1024, scene="room", views=16, mixed=True),
        # perspective training on the six faces of a cube map
        _case("graph_1m_cube6x592", "graph", 1_000_000, 592, 592, scene="polar", views=6, cube=True),
        # a roaming capture: 8 large views along a corridor, in groups of two
        _case("grouped_3m_8x4096x2048", "grouped", 3_000_000, 4096, 2048, scene="corridor", views=8, group=2),
        # the training loss on one full-size image
        _case("loss_2048x1024", "loss", 0, 2048, 1024),
        # the optimiser's step on a full-size model
        _case("adam_1m", "adam", 1_000_000, 0, 0),
        # densification of a full-size model, every few hundred steps
        _case("densify_1m", "densify", 1_000_000, 0, 0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["view", "view", "autograd", "autograd", "graph", "graph", "graph", "grouped", "loss", "adam",
                       "densify"])
    if kind in ("adam", "densify"):
        return _pure(_case("", kind, log_int(20_000, 1_500_000) | 1, 0, 0, sh=rng.choice([0, 1, 2, 3, 3])))
    if kind == "loss":
        w = log_int(200, 4096)
        return _pure(_case("", kind, 0, w, max(64, int(w * rng.uniform(0.4, 0.6)))))
    raw, sh = rng.random() < 0.4, rng.choice([0, 1, 2, 3, 3, 3])
    bg = rng.choice([0.0, 0.0, 0.5])
    log_scale = rng.uniform(-4.5, -3.5)
    if kind == "grouped":
        w = 16 * log_int(64, 192)
        return _pure(_case("", kind, log_int(200_000, 2_000_000), w, w // 2, scene=rng.choice(["corridor", "room"]),
                           sh=sh, views=rng.choice([2, 4, 6]), group=rng.choice([1, 2]), raw=raw, bg=bg,
                           log_scale=log_scale))
    n, w = log_int(1000, 1_000_000), 16 * log_int(16, 144)
    if n < 20_000:
        log_scale = rng.uniform(-3.5, -2.5)
    scene = rng.choice(["shell", "room", "smallroom", "polar"])
    if kind == "graph" and rng.random() < 0.35:
        return _pure(_case("", kind, n, 16 * log_int(8, 48), 0, scene=scene, sh=sh, views=6, cube=True, raw=raw, bg=bg,
                           log_scale=log_scale))
    views = rng.choice([1, 1, 2, 5]) if kind == "graph" else 1
    return _pure(_case("", kind, n, w, max(32, int(w * rng.uniform(0.45, 0.55))), scene=scene, sh=sh, views=views,
                       raw=raw, bg=bg, log_scale=log_scale))


def _pure(c):
    c.pop("name")
    return c


# ------------------------------------------------------------------ inputs


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device="cuda") * (hi - lo) + lo


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _box(g, n, lo, hi):
    return torch.stack([_uniform(g, n, a, b) for a, b in zip(lo, hi)], dim=1)


def _means(g, n, scene):
    if scene == "shell":  # uniform by volume between 1 m and 5 m
        d = _normal(g, n, 3)
        return d / d.norm(dim=1, keepdim=True) * (1.0 + _uniform(g, n, 0.0, 124.0)).pow(1.0 / 3.0)[:, None]
    if scene == "smallroom":
        return _box(g, n, (-5, -2, -5), (5, 2, 5))
    if scene == "room":
        return _box(g, n, (-10, -2.5, -10), (10, 2.5, 10))
    if scene == "corridor":  # 70 % uniform, 30 % in 100 clusters
        lo, hi = (0.0, -1.5, -2.0), (50.0, 1.5, 2.0)
        m = _box(g, n, lo, hi)
        centres = _box(g, 100, lo, hi)
        k = int(0.3 * n)
        if k:
            lab = torch.randint(0, 100, (k,), generator=g, device="cuda")
            c = centres[lab] + 0.3 * _normal(g, k, 3)
            m[:k] = torch.minimum(torch.maximum(c, torch.tensor(lo, device="cuda")), torch.tensor(hi, device="cuda"))
        return m[torch.randperm(n, generator=g, device="cuda")]
    # polar: 20 % within 10 degrees of the poles, 20 % within 5 degrees of the seam, 60 % in a room
    a, b = n // 5, n // 5
    y = 2.5 * _uniform(g, a, 0.0, 1.0).pow(1.0 / 3.0)
    rad = y / math.tan(math.radians(80.0)) * _uniform(g, a, 0.0, 1.0).sqrt()
    ang = _uniform(g, a, 0.0, 2.0 * math.pi)
    sign = torch.where(torch.arange(a, device="cuda") % 2 == 0, 1.0, -1.0)
    pole = torch.stack([rad * ang.cos(), sign * y, rad * ang.sin()], dim=1)
    z = 10.0 * _uniform(g, b, 0.0, 1.0).sqrt()
    seam = torch.stack([_uniform(g, b, -1.0, 1.0) * z * math.tan(math.radians(5.0)), _uniform(g, b, -2.5, 2.5), -z], dim=1)
    m = torch.cat([pole, seam, _box(g, n - a - b, (-10, -2.5, -10), (10, 2.5, 10))])
    return m[torch.randperm(n, generator=g, device="cuda")]


def _params(case, g):
    n, k = case["n"], (case["sh"] + 1) ** 2
    means = _means(g, n, case["scene"])
    log_s = case["log_scale"] + 0.7 * _normal(g, n, 3)
    quats = _normal(g, n, 4)
    logit = _normal(g, n)
    sh = 0.05 * _normal(g, n, k, 3)
    sh[:, 0] = 0.5 + 0.2 * _normal(g, n, 3)
    scales, opacity = (log_s, logit) if case["raw"] else (log_s.exp(), logit.sigmoid())
    return [t.contiguous() for t in (means, scales, quats, opacity, sh)]


def _views(case):
    w, h, nv = case["width"], case["height"], case["views"]
    if case["cube"]:
        return cubemap_views(w)
    if case["scene"] == "corridor":
        return [View.identity(w, h, (4.0 + 42.0 * i / max(nv - 1, 1), 0.0, 0.0)) for i in range(nv)]
    if nv == 1:
        return [View.identity(w, h)]
    out = []
    for i in range(nv):
        shrink = (4 if 4 * i < nv else 2 if 2 * i < nv else 1) if case["mixed"] else 1
        out.append(yaw_view(w // shrink, h // shrink, (-1.5 + 3.0 * i / (nv - 1), 0.0, 0.0), 2.399963 * i))
    return out


def _settings(case):
    return RenderSettings(sh_degree=case["sh"], raw_params=case["raw"], bg=(case["bg"],) * 3)


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    s = {"kind": kind}
    if kind == "loss":
        shape = (3, case["height"], case["width"])
        target = torch.rand(shape, generator=g, device="cuda")
        s["image"] = (target + 0.1 * _normal(g, *shape)).clamp(0.0, 1.0)
        s["target"] = target
        return s
    params = _params(case, g)
    if kind == "adam":
        s["grads"] = [1e-4 * _normal(g, *p.shape) for p in params]
        s["opt"] = GaussianAdam(params, scene_extent=10.0)
        for m, v in zip(s["opt"].m, s["opt"].v):
            m.copy_(1e-5 * _normal(g, *m.shape))
            v.copy_((1e-4 * _normal(g, *v.shape)).square() + 1e-12)
        s["opt"].t = 100
        return s
    if kind == "densify":
        # 3 % each of cloned and split Gaussians and 2 % pruned, anywhere in the arrays; whole shares, so
        # that every seed gives as many outputs
        n, stats = case["n"], D.DensifyStats(case["n"])
        order = torch.randperm(n, generator=g, device="cuda")
        k = 3 * n // 100
        clone, split, prune = order[:k], order[k:2 * k], order[2 * k:2 * k + n // 50]
        stats.count.copy_(torch.randint(0, 200, (n,), generator=g, device="cuda").to(torch.int32))
        mean = 1.9e-5 * _uniform(g, n, 0.0, 1.0)
        for hot in (clone, split):
            stats.count[hot] += 1
            mean[hot] = 1.1e-4 * _normal(g, k).abs().exp()
        stats.grad.copy_(stats.count * mean)
        stats.elev.copy_(stats.count * _uniform(g, n, 0.0, 0.9))
        params[1][clone] = params[1][clone].clamp(max=0.0199)
        params[1][split, 0] = params[1][split, 0].clamp(min=0.0201)
        params[3].clamp_(min=0.0051)
        params[3][prune] = 0.001
        s.update(params=params, stats=stats, noise=_normal(g, n, 2, 3),
                 rule=D.DensifyParams(percent_dense=1e-3, scene_extent=20.0))
        return s
    views, settings = _views(case), _settings(case)
    if kind == "view":
        s.update(params=params, views=views, settings=settings, rast=Rasterizer())
    elif kind == "autograd":
        grads = [_normal(g, 3, v.height, v.width) / (3 * v.height * v.width) for v in views]
        s.update(params=[p.requires_grad_() for p in params], views=views, settings=settings, rast=Rasterizer(),
                 grads=grads)
    else:
        targets = [torch.rand((3, v.height, v.width), generator=g, device="cuda") for v in views]
        if kind == "graph":
            s["frame"] = GraphedFrame(params, views, targets, settings)
        else:
            s["frame"] = GroupedFrame(params, views, targets, settings, group_size=case["group"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "view":
        with torch.no_grad():
            return {"images": list(render(*s["params"], s["views"], s["settings"], s["rast"]))}
    if kind == "autograd":
        images = render(*s["params"], s["views"], s["settings"], s["rast"])
        grads = torch.autograd.grad(images, s["params"], s["grads"])
        return {"images": [i.detach() for i in images], "grads": dict(zip(NAMES, grads))}
    if kind in ("graph", "grouped"):
        f = s["frame"]
        loss = f.replay() if kind == "graph" else f.step()
        return {"loss": loss, "images": list(f.images), "grads": dict(f.grads)}
    if kind == "loss":
        loss, grads = l1_dssim([s["image"]], [s["target"]])
        return {"loss": loss, "grad": grads[0]}
    if kind == "adam":
        s["opt"].step(s["grads"])
        return {"params": dict(zip(NAMES, s["opt"].params)), "m": dict(zip(NAMES, s["opt"].m)),
                "v": dict(zip(NAMES, s["opt"].v))}
    action = D.select(s["stats"], s["params"][1], s["params"][3], s["rule"])
    return {"action": action, "params": dict(zip(NAMES, D.apply(*s["params"], action, noise=s["noise"])))}


# A pixel of these scenes blends about 50 Gaussians before it stops. Per blended Gaussian the forward
# takes 23 operations (exponent 11, blend 12) and the backward 45.
BLENDS, FWD, BWD = 50, 23, 45


def work(case):
    n, kind = case["n"], case["kind"]
    floats = 11 + 3 * (case["sh"] + 1) ** 2
    if kind == "loss":
        px = 3 * case["width"] * case["height"]
        return {"bytes": 12 * px, "flops": 2 * 176 * px}  # image, target, gradient; 8 moments, 11 taps, 2 passes
    if kind == "adam":
        return {"bytes": 28 * floats * n, "flops": 12 * floats * n}
    if kind == "densify":
        return {"bytes": n * (8 * floats + 12 + 1), "flops": 20 * n}
    px = sum(v.width * v.height for v in _views(case))
    params = 4 * floats * n
    fwd = {"bytes": params + 12 * px, "flops": px * BLENDS * FWD}
    if kind == "view":
        return fwd
    # the backward reads the parameters and dL/dimage again and writes the gradients
    return {"bytes": fwd["bytes"] + 2 * params + 12 * px, "flops": fwd["flops"] + px * BLENDS * BWD}


# ------------------------------------------------------------------ the same results in 64 bits


def exact(case, seed):
    kind = case["kind"]
    if kind in ("graph", "grouped") and (case["views"] > 6 or case["n"] * case["views"] > 3_000_000):
        return None
    if case["n"] > 1_200_000 and kind not in ("adam", "densify"):
        return None
    g = _gen(seed)
    if kind == "loss":
        s = prepare(case, seed)
        loss, grad = _exact_loss(s["image"], s["target"])
        return {"loss": loss, "grad": grad}
    if kind == "adam":
        return _exact_adam(case, seed)
    if kind == "densify":
        return _exact_densify(case, seed)
    params = _params(case, g)
    views = _views(case)
    if kind == "view":
        return {"images": _exact_render(params, views, case, None)[0]}
    if kind == "autograd":
        up = [_normal(g, 3, v.height, v.width) / (3 * v.height * v.width) for v in views]
        images, grads = _exact_render(params, views, case, lambda img, i, y, x: up[i][:, y, x].double())
        return {"images": images, "grads": grads}
    targets = [torch.rand((3, v.height, v.width), generator=g, device="cuda") for v in views]

    def sign(img, i, y, x):
        return (img - targets[i][:, y, x]).sign() / (3 * views[i].height * views[i].width)

    images, grads = _exact_render(params, views, case, sign)
    loss = sum((a - t).abs().mean() for a, t in zip(images, targets))
    return {"loss": loss, "images": images, "grads": grads}


def _exact_loss(image, target, lam=0.2):
    x, y = image.double().requires_grad_(), target.double()
    _, h, w = x.shape
    k = torch.arange(-5, 6, device="cuda", dtype=torch.float64)
    k = torch.exp(-k * k / 4.5)
    k = k / k.sum()

    def blur(t):
        t = t[:, None]
        while t.shape[3] < w + 10:  # the window wraps around the seam
            grow = min(5, w) if t.shape[3] == w else 5 - min(5, w)
            t = torch.cat([t[..., -grow:], t, t[..., :grow]], dim=3)
        t = torch.nn.functional.conv2d(t, k.view(1, 1, 1, 11))
        return torch.nn.functional.conv2d(t, k.view(1, 1, 11, 1), padding=(5, 0))[:, 0]

    mx, my = blur(x), blur(y)
    sxx, syy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    ssim = (2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sxx + syy + 9e-4))
    wt = torch.sin(math.pi * (torch.arange(h, device="cuda", dtype=torch.float64) + 0.5) / h)[None, :, None]
    wt = wt / (3 * w * wt.sum())
    loss = (wt * ((1 - lam) * (x - y).abs() + lam * (1 - ssim))).sum()
    (grad,) = torch.autograd.grad(loss, x)
    return loss.detach(), grad


def _exact_adam(case, seed):
    s = prepare(case, seed)
    opt, t = s["opt"], s["opt"].t + 1
    out = {"params": {}, "m": {}, "v": {}}
    b1, b2 = opt.betas
    for name, p, gr, m, v in zip(NAMES, opt.params, s["grads"], opt.m, opt.v):
        gr, m, v = gr.double(), m.double(), v.double()
        m = b1 * m + (1 - b1) * gr
        v = b2 * v + (1 - b2) * gr * gr
        lr = opt.lr["sh_rest"] if name == "sh" else opt.lr[name]
        step = m / (1 - b1 ** t) / ((v / (1 - b2 ** t)).sqrt() + opt.eps)
        rate = torch.full_like(step, lr)
        if name == "sh":
            rate[:, 0] = opt.lr["sh_dc"]
        out["params"][name], out["m"][name], out["v"][name] = p.double() - rate * step, m, v
    return out


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], dim=1).view(-1, 3, 3)


def _exact_densify(case, seed):
    s = prepare(case, seed)
    means, scales, quats, opacity, sh = s["params"]
    r, st = s["rule"], s["stats"]
    # the decisions are stated in 32 bits, in this order of operations
    c = st.count.float()
    tau_min, tau_max = torch.tensor(r.tau_min, device="cuda"), torch.tensor(r.tau_max, device="cuda")
    hot = (st.count > 0) & (st.grad / c >= tau_min + (st.elev / c) * (tau_max - tau_min))
    big = scales.max(dim=1).values > torch.tensor(r.percent_dense, device="cuda") * torch.tensor(r.scene_extent, device="cuda")
    prune = opacity < r.min_opacity
    split, clone = hot & big & ~prune, hot & ~big & ~prune
    keep = ~prune & ~split
    action = torch.where(prune, 4, torch.where(split, 2, torch.where(clone, 1, 0))).to(torch.uint8)
    i, j, k = (m.nonzero()[:, 0] for m in (keep, clone, split))
    p64 = [p.double() for p in s["params"]]
    rot, z = _rotation(p64[2][k]), s["noise"].double()[k]
    child = [p64[0][k] + (rot @ (p64[1][k] * z[:, e]).unsqueeze(2))[..., 0] for e in (0, 1)]
    out = {}
    for name, p in zip(NAMES, p64):
        kids = child if name == "means" else [p[k] / 1.6] * 2 if name == "scales" else [p[k]] * 2
        out[name] = torch.cat([p[i], p[j]] + kids)
    return {"action": action, "params": out}


def _sh_basis(d, degree):
    x, y, z = d.unbind(1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if degree >= 1:
        c = math.sqrt(3 / (4 * pi))
        Y += [c * y, c * z, c * x]
    if degree >= 2:
        c, c0 = math.sqrt(15 / (4 * pi)), math.sqrt(5 / (16 * pi))
        Y += [c * x * y, c * y * z, c0 * (3 * z * z - 1), c * x * z, c / 2 * (x * x - y * y)]
    if degree >= 3:
        c3, c2, c1, c0 = (math.sqrt(v / pi) for v in (35 / 32, 105 / 4, 21 / 32, 7 / 16))
        Y += [c3 * y * (3 * x * x - y * y), c2 * x * y * z, c1 * y * (5 * z * z - 1), c0 * z * (5 * z * z - 3),
              c1 * x * (5 * z * z - 1), c2 / 2 * z * (x * x - y * y), c3 * x * (x * x - 3 * y * y)]
    return torch.stack(Y, dim=1)


def _project(p, v, case):
    """Per Gaussian, differentiable: u, v, the inverse covariance (3), opacity, colour (3)."""
    means, scales, quats, opacity, sh = p
    if case["raw"]:
        scales, opacity = scales.exp(), opacity.sigmoid()
    R = torch.tensor(v.R_wc, device="cuda").double()
    tr = torch.tensor(v.t_wc, device="cuda").double()
    t = means @ R.T + tr
    tx, ty, tz = t.unbind(1)
    zero = torch.zeros_like(tx)
    if v.model == 1:
        u, w = v.fx * tx / tz + v.cx, v.fy * ty / tz + v.cy
        J = torch.stack([v.fx / tz, zero, -v.fx * tx / tz ** 2, zero, v.fy / tz, -v.fy * ty / tz ** 2], 1)
    else:
        fx, fy = v.width / (2 * math.pi), v.height / math.pi
        rho2 = tx * tx + tz * tz
        rho = rho2.sqrt()
        r2 = rho2 + ty * ty
        u = fx * torch.atan2(tx, tz) + v.width / 2
        w = fy * torch.atan2(ty, rho) + v.height / 2
        J = torch.stack([fx * tz / rho2, zero, -fx * tx / rho2, -fy * tx * ty / (r2 * rho), fy * rho / r2,
                         -fy * ty * tz / (r2 * rho)], 1)
    F = J.view(-1, 2, 3) @ R @ (_rotation(quats) * scales[:, None, :])
    S = F @ F.transpose(1, 2)
    A, B, C = S[:, 0, 0] + DILATION32, S[:, 0, 1], S[:, 1, 1] + DILATION32
    det = A * C - B * B
    d = means + (R.T @ tr)
    d = d / d.norm(dim=1, keepdim=True)
    rgb = ((_sh_basis(d, case["sh"])[:, :, None] * sh).sum(1) + 0.5).clamp(min=0.0)
    return torch.cat([torch.stack([u, w, C / det, -B / det, A / det, opacity], 1), rgb], 1)


DILATION32 = float(torch.tensor(DILATION, dtype=torch.float32))


def _depth32(means, v):
    """The sorting depth, whose 32-bit order of operations is part of its definition."""
    R, tr = torch.tensor(v.R_wc, device="cuda"), torch.tensor(v.t_wc, device="cuda")
    m0, m1, m2 = means.unbind(1)
    t = [((R[i, 0] * m0 + R[i, 1] * m1) + R[i, 2] * m2) + tr[i] for i in range(3)]
    return t, t[2] if v.model == 1 else ((t[0] * t[0] + t[1] * t[1]) + t[2] * t[2]).sqrt()


def _exact_render(params, views, case, upstream):
    """Images, and with `upstream` (dL/dimage of a block of pixels) the gradients of the parameters."""
    images, total = [], [torch.zeros_like(p, dtype=torch.float64) for p in params]
    for vi, v in enumerate(views):
        t, r = _depth32(params[0], v)
        o = params[3].sigmoid() if case["raw"] else params[3]
        ok = (r > NEAR) & (r < FAR) & (255 * o > 1)
        if v.model == 1:
            u, w = v.fx * t[0].double() / t[2] + v.cx, v.fy * t[1].double() / t[2] + v.cy
            ok &= (u >= -0.3 * v.width) & (u <= 1.3 * v.width) & (w >= -0.3 * v.height) & (w <= 1.3 * v.height)
        else:
            ok &= (t[0] * t[0] + t[2] * t[2]).sqrt() > 1e-4 * r
        vis = ok.nonzero()[:, 0]
        vis = vis[torch.sort(r[vis], stable=True).indices]
        p64 = [p[vis].double().requires_grad_(upstream is not None) for p in params]
        screen = _project(p64, v, case)
        scr = screen.detach()
        det = scr[:, 2] * scr[:, 4] - scr[:, 3] ** 2
        q = 2 * torch.log(255 * scr[:, 5]) + 1e-3
        ex, ey = (q * scr[:, 4] / det).sqrt() + 1, (q * scr[:, 2] / det).sqrt() + 1
        image = torch.empty(3, v.height, v.width, dtype=torch.float64, device="cuda")
        acc = torch.zeros_like(scr)
        bw, bh = 32, 16
        for y0 in range(0, v.height, bh):
            y1 = min(y0 + bh, v.height)
            rows = ((scr[:, 1] + ey > y0) & (scr[:, 1] - ey < y1)).nonzero()[:, 0]
            ur, er = scr[rows, 0], ex[rows]
            for x0 in range(0, v.width, bw):
                x1 = min(x0 + bw, v.width)
                dc = (ur - 0.5 * (x0 + x1)).abs()
                if v.model == 0:
                    dc = torch.minimum(dc, v.width - dc)
                sel = rows[dc < er + 0.5 * (x1 - x0)]
                ys, xs = slice(y0, y1), slice(x0, x1)
                image[:, ys, xs] = _block(scr, sel, v, ys, xs, case["bg"], upstream and (
                    lambda img, ys=ys, xs=xs: upstream(img, vi, ys, xs)), acc)
        images.append(image)
        if upstream is not None:
            for full, gr in zip(total, torch.autograd.grad(screen, p64, acc)):
                full.index_add_(0, vis, gr)
    return images, dict(zip(NAMES, total))


def _block(scr, sel, v, ys, xs, bg, upstream, acc):
    """The pixels (ys, xs) from the Gaussians `sel`, in depth order; their gradients into acc."""
    E = scr[sel]
    with torch.set_grad_enabled(upstream is not None):
        E.requires_grad_(upstream is not None)
        px = torch.arange(xs.start, xs.stop, device="cuda", dtype=torch.float64) + 0.5
        py = torch.arange(ys.start, ys.stop, device="cuda", dtype=torch.float64) + 0.5
        dx = px[None, None, :] - E[:, 0, None, None]
        if v.model == 0:
            dx = dx - v.width * torch.floor(dx.detach() / v.width + 0.5)
        dy = (py[None, :] - E[:, 1, None])[:, :, None]
        power = -0.5 * (E[:, 2, None, None] * dx * dx + E[:, 4, None, None] * dy * dy) - E[:, 3, None, None] * dx * dy
        alpha = E[:, 5, None, None] * power.exp()
        alpha = torch.where(alpha >= 1.0 / 255.0, alpha.clamp(max=0.99), 0.0)
        with torch.no_grad():
            keep = torch.cumsum(torch.log1p(-alpha), 0) >= math.log(1e-4)
        alpha = torch.where(keep, alpha, 0.0)
        logs = torch.log1p(-alpha)
        behind = torch.cumsum(logs, 0)
        weight = alpha * (behind - logs).exp()
        last = logs.sum(0).exp()
        img = torch.einsum("eyx,ec->cyx", weight, E[:, 6:]) + bg * last
        if upstream is not None:
            (gr,) = torch.autograd.grad((img * upstream(img.detach())).sum(), E)
            acc.index_add_(0, sel, gr)
    return img.detach()
