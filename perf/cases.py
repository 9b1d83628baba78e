"""The work this library is asked to do, as cases that can be timed and checked.

Every case goes through the calls a user's program makes: the captured
training step (``GraphStep``), the ``torch.autograd`` entry (``rasterize``),
rendering without gradients (``Rasterizer.forward``), the photometric loss,
the parameter update and the camera global alignment. Inputs are drawn on the
GPU from a seed with the distributions of ``paper_2509_25191_gb300.synth``.

``exact`` states the same results in plain torch, in 64 bits, without the
library: projection and spherical harmonics by autograd, compositing of every
pixel over its tile's depth-sorted Gaussians.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_25191_gb300 import _lib, ga, layout
from paper_2509_25191_gb300.autograd import Rasterizer, rasterize
from paper_2509_25191_gb300.step import GraphStep

DEV = "cuda"
# the image sizes of the several-scene batch, cycled through a scene's views
LADDER = ((640, 480), (979, 546), (1237, 822), (1600, 1066))
# relative sizes of the scenes of the several-scene batch
UNEVEN = (1.0, 2.0, 4.0, 6.0, 8.0, 10.0, 12.5, 15.0)


def listed():
    def raster(name, kind, n, deg, views, v, w, h, tile, focal=1000.0, scene="cluster", scenes=1, order="given"):
        return {"name": name, "kind": kind, "n": n, "deg": deg, "scene": scene, "scenes": scenes, "views": views,
                "v": v, "w": w, "h": h, "focal": focal, "tile_w": tile[0], "tile_h": tile[1], "order": order}

    return [
        # the smallest training step: a new or tiny scene, where launches and latency are everything
        raster("step_small", "step", 2000, 0, "front", 1, 128, 128, (16, 16), focal=150.0, scene="box"),
        # the ordinary training step: one image of a grown scene per iteration
        raster("step_single_view", "step", 1_000_000, 3, "far", 1, 1237, 822, (32, 32)),
        # a batch of views of one scene in one step
        raster("step_orbit", "step", 500_000, 3, "orbit", 16, 979, 546, (32, 16)),
        # the largest: a dense scene kept in spatial order, a minibatch of large images
        raster("step_dense", "step", 6_000_000, 3, "hemisphere", 8, 1600, 1066, (32, 32), order="spatial"),
        # scenes of uneven size and images of uneven resolution in one call
        raster("step_uneven", "step", 2_600_000, 3, "orbit", 4, 0, 0, (32, 32), scenes=4),
        # a captured pose-only step: a test view's camera is tuned against frozen Gaussians
        raster("pose_tuning", "pose", 300_000, 3, "orbit", 1, 979, 546, (16, 16)),
        # a model written with torch.autograd: forward and backward of a few views, nothing captured
        raster("autograd_views", "autograd", 150_001, 2, "orbit", 3, 647, 483, (16, 16)),
        # a held-out view is rendered, no gradients, nothing captured
        raster("render_view", "render", 1_000_000, 3, "far", 1, 1600, 1066, (16, 16)),
        # the photometric loss with D-SSIM and its gradient on a batch of rendered images
        {"name": "dssim_loss", "kind": "dssim", "v": 2, "w": 1237, "h": 822, "lam": 0.2},
        # the parameter update after every step
        {"name": "adam_update", "kind": "adam", "n": 1_000_000, "deg": 3, "noise": True},
        # one iteration of the camera global alignment: 300 cameras, up to 4,096 matches a pair
        {"name": "ga_iteration", "kind": "ga_step", "cams": 300, "matches": 4096, "angle": 30.0, "ragged": False},
        # the weights and the median of the initial epipolar distances
        {"name": "ga_weights", "kind": "ga_weights", "n": 21_311_488, "bins": 100},
    ]


def draw(rng):
    def span(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("step", "step", "step", "pose", "autograd", "render", "dssim", "adam", "ga_step", "ga_weights"))
    if kind == "dssim":
        return {"kind": kind, "v": rng.randint(1, 8), "w": span(64, 1600), "h": span(48, 1066),
                "lam": rng.choice((0.2, 0.2, 0.5, 1.0))}
    if kind == "adam":
        return {"kind": kind, "n": span(2000, 6_000_000), "deg": rng.randint(0, 3), "noise": rng.random() < 0.7}
    if kind == "ga_step":
        return {"kind": kind, "cams": span(8, 300), "matches": span(100, 4096), "angle": rng.choice((30.0, 45.0)),
                "ragged": rng.random() < 0.6}
    if kind == "ga_weights":
        return {"kind": kind, "n": span(10_000, 21_000_000), "bins": rng.choice((64, 100, 100, 256))}
    views = rng.choice(("front", "far", "orbit", "hemisphere"))
    scenes = rng.choice((1, 1, 1, 2, 3)) if kind == "step" and views == "orbit" else 1
    v = {"step": rng.randint(1, 8), "pose": 1, "autograd": rng.randint(1, 4), "render": 1}[kind]
    if views in ("front", "far"):
        v = 1
    w = 0 if scenes > 1 else span(96, 1600)
    h = 0 if scenes > 1 else max(48, min(1066, int(w * rng.uniform(0.5, 1.1))))
    tile = rng.choice(((16, 16), (16, 16), (32, 16), (32, 32), (32, 32), (32, 8), (16, 8), (8, 8)))
    n = span(2000, 50_000 if views == "front" else 4_000_000 // v if v > 2 else 1_500_000)
    return {"kind": kind, "n": n, "deg": rng.randint(0, 3),
            "scene": "box" if views == "front" else "cluster", "scenes": scenes, "views": views, "v": v, "w": w, "h": h,
            "focal": 1000.0 if scenes > 1 else round(max(w, h) * rng.uniform(0.8, 1.2), 2), "tile_w": tile[0],
            "tile_h": tile[1], "order": rng.choice(("given", "spatial"))}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * (seed % 100_000_007) + 17)


def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, device=DEV)


def _rand(gen, *shape):
    return torch.rand(*shape, generator=gen, device=DEV)


def _scene(gen, n, deg, kind):
    """means, log-scales, quaternions, opacity logits, SH coefficients."""
    if kind == "box":
        means = _rand(gen, n, 3) * 2.0 - torch.tensor([1.0, 1.0, -2.0], device=DEV)
        log_scales, logits = -3.0 + 0.5 * _randn(gen, n, 3), _randn(gen, n)
    else:
        d = _randn(gen, 64, 3)
        centres = d / d.norm(dim=1, keepdim=True) * (5.0 * _rand(gen, 64, 1) ** (1.0 / 3.0))
        which = torch.randint(0, 64, (n,), generator=gen, device=DEV)
        means = centres[which] + 0.3 * _randn(gen, n, 3)
        log_scales, logits = -4.0 + 0.7 * _randn(gen, n, 3), 1.5 * _randn(gen, n)
    q = _randn(gen, n, 4)
    sh = 0.1 * _randn(gen, n, (deg + 1) ** 2, 3)
    sh[:, 0] = (_rand(gen, n, 3) - 0.5) / 0.28209479177387814
    return [means.contiguous(), log_scales, q / q.norm(dim=1, keepdim=True), logits, sh]


def _look_at(pos):
    f = -np.asarray(pos, np.float64)
    f /= np.linalg.norm(f)
    x = np.cross([0.0, 1.0, 0.0], f)
    x /= np.linalg.norm(x)
    R = np.stack([x, np.cross(f, x), f])
    return np.concatenate([R.reshape(-1), -R @ np.asarray(pos, np.float64)])


def _jitter(vm, rng, deg=1.0, frac=0.01):
    """A pose turned by deg about a random axis and moved by frac of its distance."""
    a, d = rng.standard_normal(3), rng.standard_normal(3)
    a /= np.linalg.norm(a)
    K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    th = math.radians(deg)
    R = (np.eye(3) + math.sin(th) * K + (1 - math.cos(th)) * K @ K) @ vm[:9].reshape(3, 3)
    return np.concatenate([R.reshape(-1), vm[9:] + frac * np.linalg.norm(vm[9:]) * d / np.linalg.norm(d)])


def _hemisphere(count):
    out, golden = [], math.pi * (3.0 - math.sqrt(5.0))
    for k in range(count):
        y = -(k + 0.5) / count
        r = math.sqrt(1.0 - y * y)
        out.append(_look_at((5.0 * r * math.cos(golden * k), 5.0 * y, 5.0 * r * math.sin(golden * k))))
    return out


def _ladder(scene, v):
    """The image sizes of a scene's views in the several-scene batch."""
    return [LADDER[(scene + k) % len(LADDER)] for k in range(v)]


def _cameras(case, seed, scene):
    """viewmats [V,12], width, height of one scene's views."""
    rng = np.random.default_rng(seed * 16 + scene)
    v = case["v"]
    if case["views"] == "front":
        mats = [np.concatenate([np.eye(3).reshape(-1), np.zeros(3)])]
    elif case["views"] == "far":
        mats = [_look_at((0.0, 0.0, -6.0))]
    elif case["views"] == "orbit":
        th = rng.uniform(0, 2 * math.pi) + 2 * math.pi * np.arange(v) / v
        mats = [_look_at((5.0 * math.sin(t), 0.0, -5.0 * math.cos(t))) for t in th]
    else:
        every = _hemisphere(300)
        mats = [every[k] for k in rng.choice(300, v, replace=False)]
    mats = np.stack([_jitter(m, rng) for m in mats])
    if case["scenes"] > 1:
        size = _ladder(scene, v)
        return mats, [w for w, _ in size], [h for _, h in size]
    return mats, [case["w"]] * v, [case["h"]] * v


def _photo(gen, width, height):
    """Target images: smooth patterns with some noise, in [0, 1], views one after another."""
    out = []
    for w, h in zip(width, height):
        x = torch.arange(w, device=DEV) / 200.0
        y = torch.arange(h, device=DEV)[:, None] / 200.0
        k = 6.0 * _randn(gen, 3, 4, 2)
        ph = 6.3 * _rand(gen, 3, 4)
        img = 0.5 + 0.12 * sum(torch.sin(k[:, i, 0, None, None] * x + k[:, i, 1, None, None] * y + ph[:, i, None, None])
                               for i in range(4))
        out.append((img + 0.05 * _randn(gen, 3, h, w)).clamp(0.0, 1.0).reshape(-1))
    return torch.cat(out)


def _raster_inputs(case, seed):
    gen = _gen(seed)
    S = case["scenes"]
    weights = UNEVEN[:S]
    sizes = [max(1, int(case["n"] * x / sum(weights))) for x in weights]
    parts = [_scene(gen, n, case["deg"], case["scene"]) for n in sizes]
    params = [torch.cat(p).contiguous() if S > 1 else p[0] for p in zip(*parts)]
    mats, width, height, begin, count, at = [], [], [], [], [], 0
    for s, n in enumerate(sizes):
        m, w, h = _cameras(case, seed, s)
        mats.append(m)
        width += w
        height += h
        begin += [at] * len(w)
        count += [n] * len(w)
        at += n
    if case["order"] == "spatial":
        starts = np.cumsum([0] + sizes[:-1])
        perm = layout.spatial_order(params[0], list(zip(starts, sizes)))
        params = [p.index_select(0, perm).contiguous() for p in params]
    vm = torch.as_tensor(np.concatenate(mats).astype(np.float32)).to(DEV)
    intr = torch.tensor([[case["focal"], case["focal"], w / 2.0, h / 2.0] for w, h in zip(width, height)], device=DEV)
    return params, vm, intr, width, height, begin, count, _photo(gen, width, height)


def _ga_inputs(case, seed):
    """True and initial cameras on a hemisphere, the pairs whose viewing
    directions are close, and noisy matches of random scene points."""
    gen, rng, n = _gen(seed), np.random.default_rng(seed), case["cams"]
    true = np.stack(_hemisphere(n))
    vm0 = np.stack([_jitter(m, rng) for m in true]).astype(np.float32)
    intr = np.tile([1000.0, 1000.0, 800.0, 533.0], (n, 1))
    intr0 = intr.copy()
    intr0[:, :2] *= 1.0 + rng.uniform(-0.02, 0.02, (n, 1))
    d = vm0[:, 6:9].astype(np.float64)
    i, j = np.nonzero(np.triu(d @ d.T > math.cos(math.radians(case["angle"])), 1))
    if len(i) == 0:
        i, j = np.array([0]), np.array([1])
    per = np.full(len(i), case["matches"], np.int64)
    if case["ragged"]:
        per = rng.integers(0, case["matches"] + 1, len(i))
    offsets = np.concatenate([[0], np.cumsum(per)])
    to = lambda a: torch.as_tensor(a).to(DEV)
    pair = torch.repeat_interleave(torch.arange(len(i), device=DEV), to(per))
    K = pair.shape[0]
    p = _randn(gen, K, 3)
    p = p / p.norm(dim=1, keepdim=True) * (2.0 * _rand(gen, K, 1) ** (1.0 / 3.0))
    tv = to(true.astype(np.float32))
    uv = []
    for cam in (to(i)[pair], to(j)[pair]):
        c = torch.einsum("kab,kb->ka", tv[cam, :9].reshape(-1, 3, 3), p) + tv[cam, 9:]
        uv.append(1000.0 * c[:, :2] / c[:, 2:] + torch.tensor([800.0, 533.0], device=DEV) + 0.5 * _randn(gen, K, 2))
    out = _rand(gen, K, 1) < 0.15
    uv[1] = torch.where(out, _rand(gen, K, 2) * torch.tensor([1600.0, 1066.0], device=DEV), uv[1])
    return (to(intr0.astype(np.float32)), to(vm0), to(np.stack([i, j], 1).astype(np.int32)), to(offsets),
            torch.cat(uv, 1).contiguous())


def _adam_inputs(case, seed):
    """(params, grads, first and second moments, learning rates, noise) of the five parameter arrays."""
    gen = _gen(seed)
    params = _scene(gen, case["n"], case["deg"], "cluster")
    grads = [1e-6 * _randn(gen, *p.shape) for p in params]
    m = [1e-6 * _randn(gen, *p.shape) for p in params]
    v = [1e-12 * _rand(gen, *p.shape) for p in params]
    noise = _randn(gen, case["n"], 3) if case["noise"] else None
    return params, grads, m, v, (1.6e-4, 5e-3, 1e-3, 5e-2, 2.5e-3), noise


def _dssim_inputs(case, seed):
    gen, w, h = _gen(seed), [case["w"]] * case["v"], [case["h"]] * case["v"]
    target = _photo(gen, w, h)
    return (target + 0.1 * _randn(gen, target.numel())).clamp_(0.0, 1.0), target, w, h


def _distances(case, seed):
    """Epipolar distances in pixels: most are a few pixels, the outliers up to hundreds."""
    gen, n = _gen(seed), case["n"]
    e = (6.0 * _randn(gen, n)).abs()
    return torch.where(_rand(gen, n) < 0.15, 700.0 * _rand(gen, n), e)


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "dssim":
        image, target, w, h = _dssim_inputs(case, seed)
        z = np.zeros(len(w), np.int64)
        return {"kind": kind, "image": image, "target": target, "views": _lib.Views(None, None, w, h, z, z),
                "loss": torch.empty(3, device=DEV), "grad": torch.empty_like(image), "lam": case["lam"]}
    if kind == "adam":
        params, grads, m, v, lrs, noise = _adam_inputs(case, seed)
        return {"kind": kind, "groups": list(zip(params, grads, m, v, lrs)), "noise": noise, "step": 100}
    if kind == "ga_step":
        intr0, vm0, pairs, offsets, matches = _ga_inputs(case, seed)
        al = ga.GlobalAlignment(intr0, vm0, pairs, offsets, matches)
        return {"kind": kind, "ga": al, "d_res": torch.empty(al.n, 10, device=DEV)}
    if kind == "ga_weights":
        return {"kind": kind, "dist": _distances(case, seed), "bins": case["bins"]}
    params, vm, intr, width, height, begin, count, target = _raster_inputs(case, seed)
    tile = (case["tile_w"], case["tile_h"])
    if kind in ("step", "pose"):
        views = _lib.Views(vm, intr, width, height, begin, count)
        step = GraphStep(_lib.Gaussians(*params), views, target, tile=tile,
                         want_gaussian_grads=kind == "step")
        return {"kind": kind, "step": step}
    rast = Rasterizer(tile=tile)
    if kind == "render":
        return {"kind": kind, "rast": rast, "g": _lib.Gaussians(*params),
                "views": _lib.Views(vm, intr, width, height, begin, count)}
    leaves = [t.requires_grad_(True) for t in params + [vm]]
    return {"kind": kind, "rast": rast, "leaves": leaves, "intr": intr, "size": (width, height), "target": target}


def run(s):
    kind = s["kind"]
    if kind in ("step", "pose"):
        st = s["step"]
        st.replay()
        out = [st.image, st.loss, st.dviewmat, st.dtwist]
        g = st.grads
        return out + [g.means, g.log_scales, g.quats, g.opacity_logits, g.sh] if kind == "step" else out
    if kind == "render":
        image, _ = s["rast"].forward(s["g"], s["views"])
        return [image]
    if kind == "autograd":
        image = rasterize(*s["leaves"], s["intr"], *s["size"], rasterizer=s["rast"])
        loss = (image - s["target"]).square().mean()
        return [image.detach(), loss.detach(), *torch.autograd.grad(loss, s["leaves"])]
    if kind == "dssim":
        _lib.gs_l1_dssim_loss(s["views"], s["image"], s["target"], s["loss"], s["grad"], s["lam"])
        return [s["loss"], s["grad"]]
    if kind == "adam":
        s["step"] += 1
        _lib.gs_sgld_adam_step(s["groups"], s["step"], noise=s["noise"], noise_scale=1e-5 if s["noise"] is not None else 0.0)
        return [t for grp in s["groups"] for t in (grp[0], grp[2], grp[3])]
    if kind == "ga_step":
        loss = s["ga"].step(s["d_res"])
        return [loss, s["d_res"], s["ga"].res, s["ga"].res_m, s["ga"].res_v, s["ga"].vm, s["ga"].intr]
    weights, counts, stats = ga.pdf_weights(s["dist"], s["bins"])
    return [weights, counts, stats]


def work(case):
    kind = case["kind"]
    K = (case.get("deg", 0) + 1) ** 2
    row = 4 * (11 + 3 * K)                       # bytes of one Gaussian's parameters
    if kind == "dssim":
        px = 3 * case["v"] * case["w"] * case["h"]
        return {"bytes": 12 * px, "flops": 2 * 11 * 2 * 8 * px}      # 8 separable 11-tap blurs
    if kind == "adam":
        return {"bytes": case["n"] * (7 * row + (12 if case["noise"] else 0)), "flops": 14 * case["n"] * row / 4}
    if kind == "ga_step":
        # viewing directions on the hemisphere: the share of pairs within the angle
        n = case["cams"]
        pairs = max(1.0, n * (n - 1) / 2 * (1 - math.cos(math.radians(case["angle"]))) * 0.87)
        k = pairs * case["matches"] * (0.5 if case["ragged"] else 1.0)
        return {"bytes": 20 * k + 64 * n, "flops": 60 * k}
    if kind == "ga_weights":
        return {"bytes": 8 * case["n"], "flops": 4 * case["n"]}
    if case["scenes"] > 1:
        px = sum(w * h for s in range(case["scenes"]) for w, h in _ladder(s, case["v"]))
    else:
        px = case["v"] * case["w"] * case["h"]
    slots = case["n"] * case["v"]
    if kind == "render":
        return {"bytes": case["n"] * row + 12 * px, "flops": 300 * slots + 12 * 100 * px}
    grads = 1 if kind == "pose" else 2
    # parameters in, their gradients out, target in, image out; about a hundred
    # Gaussians reach a pixel before it is opaque
    return {"bytes": grads * case["n"] * row + 24 * px, "flops": 900 * slots + 52 * 100 * px}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind == "dssim":
        return _exact_dssim(*_dssim_inputs(case, seed), case["lam"])
    if kind == "adam":
        return _exact_adam(*_adam_inputs(case, seed))
    if kind == "ga_step":
        return _exact_ga_step(*_ga_inputs(case, seed))
    if kind == "ga_weights":
        return _exact_weights(_distances(case, seed), case["bins"])
    if case["n"] * case["v"] > 11_000_000:
        return None                              # (about a minute)
    return _exact_raster(case, seed)


def _exact_adam(params, grads, m, v, lrs, noise):
    out, t, b1, b2 = [], 101, 0.9, 0.999
    for k, (p, g, a, b, lr) in enumerate(zip(params, grads, m, v, lrs)):
        g = g.double()
        a, b = b1 * a.double() + (1 - b1) * g, b2 * b.double() + (1 - b2) * g * g
        p = p.double() - lr * (a / (1 - b1 ** t)) / ((b / (1 - b2 ** t)).sqrt() + 1e-15)
        if k == 0 and noise is not None:
            p = p + 1e-5 * noise.double()
        out += [p, a, b]
    return out


def _exact_dssim(image, target, width, height, lam):
    win = torch.exp(-torch.arange(-5, 6, device=DEV, dtype=torch.float64) ** 2 / 4.5)
    win = win / win.sum()

    def blur(t):
        t = torch.nn.functional.conv2d(t, win.view(1, 1, 1, 11), padding=(0, 5))
        return torch.nn.functional.conv2d(t, win.view(1, 1, 11, 1), padding=(5, 0))

    x, y = image.double().requires_grad_(True), target.double()
    l1, ssim, at = 0.0, 0.0, 0
    for w, h in zip(width, height):
        a, b = (t[at:at + 3 * w * h].view(3, 1, h, w) for t in (x, y))
        mu, nu = blur(a), blur(b)
        saa, sbb, sab = blur(a * a) - mu * mu, blur(b * b) - nu * nu, blur(a * b) - mu * nu
        ssim = ssim + ((2 * mu * nu + 1e-4) * (2 * sab + 9e-4) / ((mu * mu + nu * nu + 1e-4) * (saa + sbb + 9e-4))).sum()
        l1 = l1 + (a - b).abs().sum()
        at += 3 * w * h
    l1, ds = l1 / at, 1 - ssim / at
    loss = (1 - lam) * l1 + lam * ds
    grad, = torch.autograd.grad(loss, x)
    return [torch.stack([loss, l1, ds]).detach(), grad]


def _exact_weights(dist, bins):
    # the bin of a distance is defined by its float32 product
    inv = torch.tensor(float(bins), device=DEV) / dist.max()
    at = (dist * inv).floor().clamp(0, bins - 1).long()
    counts = torch.bincount(at, minlength=bins).double()
    table = (dist.numel() * counts / counts.square().sum()).sqrt()
    order = dist.sort().values.double()
    n = dist.numel()
    stats = torch.stack([order[-1], order[(n - 1) // 2], order[n // 2], torch.zeros((), device=DEV, dtype=torch.float64)])
    return [table[at], None, stats]


def _rotation_6d(r):
    b1 = r[:, :3] / r[:, :3].norm(dim=1, keepdim=True)
    b2 = r[:, 3:] - (b1 * r[:, 3:]).sum(1, keepdim=True) * b1
    b2 = b2 / b2.norm(dim=1, keepdim=True)
    return torch.stack([b1, b2, torch.cross(b1, b2, dim=1)], dim=2)


def _exact_ga_step(intr0, vm0, pairs, offsets, matches):
    n = intr0.shape[0]
    intr0, vm0, pairs = intr0.double(), vm0.double(), pairs.long()
    pair = torch.repeat_interleave(torch.arange(pairs.shape[0], device=DEV), offsets[1:] - offsets[:-1])

    def geometry(intr, vm):
        R, t = vm[:, :9].reshape(-1, 3, 3), vm[:, 9:]
        K = torch.zeros(n, 3, 3, device=DEV, dtype=torch.float64)
        K[:, 0, 0], K[:, 1, 1] = 1 / intr[:, 0], 1 / intr[:, 1]
        K[:, 0, 2], K[:, 1, 2], K[:, 2, 2] = -intr[:, 2] / intr[:, 0], -intr[:, 3] / intr[:, 1], 1.0
        i, j = pairs.T
        Rij = R[j] @ R[i].transpose(1, 2)
        tij = t[j] - (Rij @ t[i][:, :, None])[:, :, 0]
        X = torch.zeros(len(i), 3, 3, device=DEV, dtype=torch.float64)
        X[:, 0, 1], X[:, 0, 2], X[:, 1, 2] = -tij[:, 2], tij[:, 1], -tij[:, 0]
        X[:, 1, 0], X[:, 2, 0], X[:, 2, 1] = tij[:, 2], -tij[:, 1], tij[:, 0]
        return K[j].transpose(1, 2) @ X @ Rij @ K[i]

    def distances(F, at, stop):
        q, f = matches[at:stop].double(), F[pair[at:stop]]
        line = f[:, :, 0] * q[:, 0:1] + f[:, :, 1] * q[:, 1:2] + f[:, :, 2]
        return (line[:, 0] * q[:, 2] + line[:, 1] * q[:, 3] + line[:, 2]).abs() / line[:, :2].norm(dim=1)

    chunk, total = 2_000_000, matches.shape[0]
    F0 = geometry(intr0, vm0)
    e0 = torch.cat([distances(F0, k, min(total, k + chunk)) for k in range(0, total, chunk)]) if total else matches.new_zeros(0).double()
    w, _, st = _exact_weights(e0.float(), 100) if total else (e0, None, torch.zeros(4, dtype=torch.float64, device=DEV))
    w = w.double()
    lr = 5e-4 if float(st[1] + st[2]) / 2 < 2.5 else 1e-2 if float(st[1] + st[2]) / 2 > 7.5 else 1e-3
    res = torch.zeros(n, 10, device=DEV, dtype=torch.float64)
    res[:, 0] = res[:, 4] = 1.0
    res.requires_grad_(True)
    vm = torch.cat([(_rotation_6d(res[:, :6]) @ vm0[:, :9].reshape(-1, 3, 3)).reshape(-1, 9), vm0[:, 9:] + res[:, 6:9]], 1)
    intr = torch.cat([intr0[:, :2] * torch.exp(res[:, 9:]), intr0[:, 2:]], 1)
    F = geometry(intr, vm)
    leaf, loss = F.detach().requires_grad_(True), torch.zeros(1, device=DEV, dtype=torch.float64)
    gF, W = torch.zeros_like(leaf), w.sum().clamp(min=1e-300)
    for k in range(0, total, chunk):
        part = (distances(leaf, k, min(total, k + chunk)) * w[k:k + chunk]).sum() / W
        gF += torch.autograd.grad(part, leaf)[0]
        loss += part.detach()
    g, = torch.autograd.grad(F, res, gF)
    m, v = 0.1 * g, 0.001 * g * g
    new = res.detach() - lr * (m / 0.1) / ((v / 0.001).sqrt() + 1e-15)
    return [loss, g, new, m, v, vm.detach(), intr.detach()]


def _sh_basis(deg, d):
    """Real spherical harmonics with the Condon-Shortley phase, index l*l + l + m."""
    x, y, z = d.unbind(1)
    re, im = [torch.ones_like(x)], [torch.zeros_like(x)]
    for _ in range(deg):
        re, im = re + [re[-1] * x - im[-1] * y], im + [re[-1] * y + im[-1] * x]
    # m-th derivatives of the Legendre polynomials
    one = torch.ones_like(z)
    P = {(0, 0): one, (1, 0): z, (1, 1): one, (2, 0): (3 * z * z - 1) / 2, (2, 1): 3 * z, (2, 2): 3 * one,
         (3, 0): (5 * z ** 3 - 3 * z) / 2, (3, 1): (15 * z * z - 3) / 2, (3, 2): 15 * z, (3, 3): 15 * one}
    out = []
    for l in range(deg + 1):
        for m in range(-l, l + 1):
            a = abs(m)
            k = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - a) / math.factorial(l + a))
            k *= (math.sqrt(2.0) if a else 1.0) * (-1) ** a
            out.append(k * P[l, a] * (im[a] if m < 0 else re[a]))
    return torch.stack(out, 1)


def _exact_project(p, vm, intr, w, h, deg):
    """Per Gaussian: (mean [n,2], dilated covariance (a, b, c) [n,3], opacity, colour),
    then without gradient depth (float32), reach [n,2], radius, visible."""
    mu, ls, q, lg, sh = p
    R, t = vm[:9].reshape(3, 3), vm[9:]
    fx, fy, cx, cy = intr.double().tolist()
    x, y, z = (mu @ R.T + t).unbind(1)
    q = q / q.norm(dim=1, keepdim=True)
    a, b, c, d = q.unbind(1)
    Rq = torch.stack([1 - 2 * (c * c + d * d), 2 * (b * c - a * d), 2 * (b * d + a * c),
                      2 * (b * c + a * d), 1 - 2 * (b * b + d * d), 2 * (c * d - a * b),
                      2 * (b * d - a * c), 2 * (c * d + a * b), 1 - 2 * (b * b + c * c)], 1).reshape(-1, 3, 3)
    M = Rq * torch.exp(ls)[:, None, :]
    lx, ly = 1.3 * 0.5 * w / fx, 1.3 * 0.5 * h / fy
    u, v = (x / z).clamp(-lx, lx), (y / z).clamp(-ly, ly)
    J0 = torch.stack([fx / z, torch.zeros_like(z), -fx * u / z], 1) @ R
    J1 = torch.stack([torch.zeros_like(z), fy / z, -fy * v / z], 1) @ R
    r0, r1 = (J0[:, None] @ M)[:, 0], (J1[:, None] @ M)[:, 0]
    cov = torch.stack([(r0 * r0).sum(1) + 0.3, (r0 * r1).sum(1), (r1 * r1).sum(1) + 0.3], 1)
    mean = torch.stack([fx * x / z + cx, fy * y / z + cy], 1)
    o = torch.sigmoid(lg)
    d = mu + R.T @ t
    col = torch.einsum("nk,nkc->nc", _sh_basis(deg, d / d.norm(dim=1, keepdim=True)), sh) + 0.5
    with torch.no_grad():
        det, mid = cov[:, 0] * cov[:, 2] - cov[:, 1] ** 2, 0.5 * (cov[:, 0] + cov[:, 2])
        radius = torch.ceil(3 * (mid + (mid * mid - det).clamp(min=0.1).sqrt()).sqrt())
        k = 2 * torch.log(o * 255.0)
        vis = (z > 0.2) & (det > 0) & (k > 0) & (mean[:, 0] + radius >= 0) & (mean[:, 0] - radius <= w) & \
            (mean[:, 1] + radius >= 0) & (mean[:, 1] - radius <= h)
        reach = torch.minimum((k.clamp(min=0)[:, None] * cov[:, ::2]).sqrt(), radius[:, None])
    return (mean, cov, o, col.clamp(min=0)), z.detach().float(), reach, radius, vis


def _tile_chunks(mean, reach, depth, w, h, side=16, budget=24_000_000):
    """Tiles in groups of similar list length: (tile ids [t], Gaussians in
    depth order [t, L], -1 past a list's end)."""
    gx, gy = -(-w // side), -(-h // side)
    ids = torch.sort(depth, stable=True).indices
    lo = torch.floor((mean[ids] - reach[ids]) / side).clamp(min=0)
    hi = torch.floor((mean[ids] + reach[ids]) / side) + 1
    lim = torch.tensor([gx, gy], device=DEV, dtype=lo.dtype)
    lo, hi = torch.minimum(lo, lim).long(), torch.minimum(hi.clamp(min=0), lim).long()
    span = (hi - lo).clamp(min=0)
    per = span[:, 0] * span[:, 1]
    own = torch.repeat_interleave(torch.arange(len(ids), device=DEV), per)
    at = torch.arange(len(own), device=DEV) - (torch.cumsum(per, 0) - per)[own]
    sx = span[own, 0]
    tile = (lo[own, 1] + at // sx.clamp(min=1)) * gx + lo[own, 0] + at % sx.clamp(min=1)
    tile, order = torch.sort(tile, stable=True)
    own = ids[own[order]]
    count = torch.bincount(tile, minlength=gx * gy)
    first = torch.cumsum(count, 0) - count
    by = torch.sort(count, descending=True).indices
    lens, k = count[by].tolist(), 0
    while k < len(lens) and lens[k] > 0:
        t = max(1, min(len(lens) - k, budget // (lens[k] * side * side)))
        tiles = by[k:k + t]
        j = torch.arange(lens[k], device=DEV)[None]
        inside = j < count[tiles][:, None]
        src = (first[tiles][:, None] + j).clamp(max=len(own) - 1)
        yield tiles, torch.where(inside, own[src], -1)
        k += t


def _composite(tiles, lists, two_d, radius, w, side=16):
    """[t, 3, side*side] colours of the tiles' pixels."""
    gx = -(-w // side)
    mean, cov, o, col = two_d
    k, pad = lists.clamp(min=0), lists < 0
    px = torch.arange(side, device=DEV, dtype=torch.float64) + 0.5
    X = ((tiles % gx) * side)[:, None] + px.repeat(side)
    Y = ((tiles // gx) * side)[:, None] + px.repeat_interleave(side)
    m, s, r = mean[k], cov[k], radius[k]
    dx, dy = X[:, None] - m[:, :, :1], Y[:, None] - m[:, :, 1:]
    a, b, c = s[:, :, :1], s[:, :, 1:2], s[:, :, 2:]
    power = -0.5 * (c * dx * dx - 2 * b * dx * dy + a * dy * dy) / (a * c - b * b)
    alpha = (o[k][:, :, None] * torch.exp(power)).clamp(max=0.99)
    ok = (alpha >= 1.0 / 255.0) & (dx.abs() <= r[:, :, None]) & (dy.abs() <= r[:, :, None]) & ~pad[:, :, None]
    log1 = torch.where(ok, torch.log1p(-alpha), torch.zeros((), device=DEV, dtype=torch.float64))
    after = torch.cumsum(log1, 1)
    keep = ok & (after.detach() >= math.log(1e-4))
    weight = torch.where(keep, alpha * torch.exp(after - log1), torch.zeros((), device=DEV, dtype=torch.float64))
    return torch.einsum("tlp,tlc->tcp", weight, col[k])


def _exact_raster(case, seed):
    params, vm, intr, width, height, begin, count, target = _raster_inputs(case, seed)
    kind, deg, side = case["kind"], case["deg"], 16
    total = sum(3 * w * h for w, h in zip(width, height))
    image, grads = [], [torch.zeros_like(p, dtype=torch.float64) for p in params]
    dvm, loss, base = torch.zeros_like(vm, dtype=torch.float64), 0.0, 0
    for v, (w, h) in enumerate(zip(width, height)):
        lo, hi = begin[v], begin[v] + count[v]
        pose = vm[v].double()
        with torch.no_grad():
            seen = _exact_project([p[lo:hi].double() for p in params], pose, intr[v], w, h, deg)[-1]
        seen = lo + torch.nonzero(seen)[:, 0]
        leaf = [p[seen].double().requires_grad_(kind != "render") for p in params] + [pose.requires_grad_(kind != "render")]
        full, depth, reach, radius, _ = _exact_project(leaf[:5], pose, intr[v], w, h, deg)
        two_d = [t.detach().requires_grad_(kind != "render") for t in full]
        gx, gy = -(-w // side), -(-h // side)
        img = torch.zeros(gx * gy, 3, side * side, device=DEV, dtype=torch.float64)
        tgt = torch.zeros(3, gy * side, gx * side, device=DEV, dtype=torch.float64)
        tgt[:, :h, :w] = target[base:base + 3 * w * h].view(3, h, w)
        inside = torch.zeros(1, gy * side, gx * side, device=DEV, dtype=torch.float64)
        inside[:, :h, :w] = 1.0
        tiled = lambda t: t.view(-1, gy, side, gx, side).permute(1, 3, 0, 2, 4).reshape(gx * gy, -1, side * side)
        tgt, inside = tiled(tgt), tiled(inside)
        acc = [torch.zeros_like(t) for t in two_d]
        for tiles, lists in _tile_chunks(two_d[0].detach(), reach, depth, w, h):
            out = _composite(tiles, lists, two_d, radius, w)
            img[tiles] = out.detach()
            if kind != "render":
                diff = (out.detach() - tgt[tiles]) * inside[tiles]
                up = torch.sign(diff) / total if kind != "autograd" else 2 * diff / total
                for s, g in zip(acc, torch.autograd.grad(out, two_d, up)):
                    s += g
        diff = (img - tgt) * inside
        loss += float((diff.abs() if kind != "autograd" else diff.square()).sum()) / total
        flat = img.view(gy, gx, 3, side, side).permute(2, 0, 3, 1, 4).reshape(3, gy * side, gx * side)
        image.append(flat[:, :h, :w].reshape(-1))
        if kind != "render":
            got = torch.autograd.grad(full, leaf, acc)
            for s, g in zip(grads, got):
                s.index_add_(0, seen, g)
            dvm[v] += got[-1]
        base += 3 * w * h
    image = torch.cat(image)
    if kind == "render":
        return [image]
    loss = torch.tensor([loss], device=DEV, dtype=torch.float64)
    if kind == "autograd":
        return [image, loss.reshape(()), *grads, dvm]
    R, t, gR, gt = vm[:, :9].double().reshape(-1, 3, 3), vm[:, 9:].double(), dvm[:, :9].reshape(-1, 3, 3), dvm[:, 9:]
    A = gR @ R.transpose(1, 2) + gt[:, :, None] * t[:, None, :]
    twist = torch.cat([gt, torch.stack([A[:, 2, 1] - A[:, 1, 2], A[:, 0, 2] - A[:, 2, 0], A[:, 1, 0] - A[:, 0, 1]], 1)], 1)
    out = [image, loss, dvm, twist]
    return out + grads if kind == "step" else out
