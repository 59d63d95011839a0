"""The work this framework is used for, as cases that can be timed and compared.

A case renders a Level-of-Detail Gaussian tree through the public binding
(``paper_2603_23891_gb300.filtergs``).  The trees follow the recipes of ``synth``
(the uniform box, the blob field, the city), drawn and built on the GPU so that
10M leaves take seconds.  What a seed draws is what changes from call to call in
real use: the camera poses and, for the differentiable form, the parameters and
the target image.  The loaded tree is kept per case, as a program that renders
many poses of one scene keeps it.

A case's fields: kind (what is called), scene / leaves / degree (the tree and its
SH degree), width x height (the image), views, tile_w x tile_h, tau_R (the LoD
threshold in pixels) and tau (the shrinking threshold, 0 for the 3-sigma
footprint).
"""
import math
from functools import lru_cache
from types import SimpleNamespace

import numpy as np
import torch

from paper_2603_23891_gb300 import filtergs, synth

PARAMS = filtergs.GRAD_FIELDS


def listed():
    def case(name, kind, scene, leaves, degree, width, height, views=1, tile=(16, 16), tau_R=3.0, tau=0.0):
        return dict(name=name, kind=kind, scene=scene, leaves=leaves, degree=degree, width=width, height=height,
                    views=views, tile_w=tile[0], tile_h=tile[1], tau_R=tau_R, tau=tau)

    return [
        # a thumbnail of a small object: launches and latency
        case("frame-tiny", "frame", "box", 4096, 0, 256, 256, tau_R=1.0),
        # a preview window of a middling scene, ragged on both sides, the wide tile shape
        case("frame-preview", "frame", "blobs", 60_000, 1, 803, 601, tile=(32, 8)),
        # an interactive frame before calibration: the 3-sigma footprint, at 1080p
        case("frame-blobs", "frame", "blobs", 1_000_000, 3, 1920, 1080),
        # the flythrough frame: the 10M-leaf city at 1080p with adaptive shrinking
        case("frame-city", "frame", "city", 10_000_000, 3, 1920, 1080, tau=0.0772),
        # the same at 4K, odd by a pixel each way
        case("frame-city-4k", "frame", "city", 10_000_000, 3, 3839, 2159, tau=0.0772),
        # serving: every frame into pinned host memory, the copy behind the next frame
        case("serve-city", "serve", "city", 2_000_000, 3, 1920, 1080, tau=0.0772),
        # many viewers at once: views of 640 to 3840 columns in one call
        case("batch-city", "batch", "city", 10_000_000, 3, 1920, 1080, views=8, tau=0.0772),
        # one training step: parameters in, image and gradients out, through autograd
        case("train-small", "train", "blobs", 20_000, 2, 400, 301),
        case("train-blobs", "train", "blobs", 1_000_000, 3, 1920, 1080),
        # gradients of several views added up, transmittance recomputed
        case("accumulate", "accumulate", "blobs", 300_000, 3, 960, 540, views=2, tau=0.02),
        # scene calibration: the KPC / GTC pre-render of a handful of views
        case("calibrate", "calibrate", "blobs", 1_000_000, 3, 1920, 1080, views=4),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["frame", "frame", "frame", "serve", "batch", "train", "accumulate", "calibrate"])
    learning = kind in ("train", "accumulate")
    scene = rng.choice(["box", "blobs"] if learning else ["box", "blobs", "city"])
    width = spread(200, 1920 if learning or kind in ("batch", "calibrate") else 3840)
    tile = rng.choice([(16, 16), (16, 16), (32, 8), (8, 32)])
    return dict(kind=kind, scene=scene, leaves=spread(2000, 20_000 if scene == "box" else 1_000_000 if learning else 3_000_000),
                degree=rng.randrange(4), width=width, height=max(120, int(width * rng.uniform(0.5, 0.8))),
                views=1 if kind in ("frame", "serve", "train") else rng.randrange(2, 7), tile_w=tile[0], tile_h=tile[1],
                tau_R=round(rng.uniform(1.0, 6.0), 2), tau=rng.choice([0.0, round(rng.uniform(1 / 255, 0.15), 4)]))


# ---------------------------------------------------------------- scenes
def _leaves(scene, n, gen):
    """Leaf centres, mean and spread of the log-scales and of the opacity logits."""
    dev = torch.device("cuda")

    def uniform(lo, hi, *shape):
        return torch.rand(*shape, generator=gen, device=dev) * (hi - lo) + lo

    if scene == "box":
        mu = uniform(-1, 1, n, 3) * torch.tensor([32.0, 32.0, 4.0], device=dev)
        return mu, (-1.5, 0.3), (0.0, 1.0)
    if scene == "blobs":
        lo, hi = torch.tensor([-250.0, -250.0, 0.0], device=dev), torch.tensor([250.0, 250.0, 50.0], device=dev)
        centre, sigma = uniform(0, 1, 2000, 3) * (hi - lo) + lo, uniform(2.0, 20.0, 2000)
        b = torch.randint(0, 2000, (n,), generator=gen, device=dev)
        mu = centre[b] + torch.randn(n, 3, generator=gen, device=dev) * sigma[b, None]
        out = (mu < lo) | (mu > hi)               # folded back into the box
        return torch.where(out, uniform(0, 1, n, 3) * (hi - lo) + lo, mu), (-2.0, 0.5), (0.0, 1.5)
    boxes = 5000
    size = torch.stack([uniform(10, 60, boxes), uniform(10, 60, boxes), uniform(5, 80, boxes)], 1)
    at = torch.cat([uniform(-970, 970, boxes, 2), torch.zeros(boxes, 1, device=dev)], 1)
    w, d, h = size.unbind(1)
    area = torch.stack([d * h, d * h, w * h, w * h, w * d], 1).flatten().double().cumsum(0).cpu()
    pick = torch.searchsorted((area / area[-1]).to(dev), torch.rand(n, generator=gen, device=dev).double()).clamp_(max=5 * boxes - 1)
    b, face = pick // 5, pick % 5
    p = uniform(-0.5, 0.5, n, 3)                  # in the unit box, z over [0, 1]
    p[:, 2] += 0.5
    for axis in (0, 1):
        for side in (0, 1):
            p[face == 2 * axis + side, axis] = 0.5 - side
    p[face == 4, 2] = 1.0
    mu = at[b] + p * size[b]
    ground = torch.rand(n, generator=gen, device=dev) < 0.3
    flat = torch.cat([uniform(-1000, 1000, n, 2), 0.5 * torch.randn(n, 1, generator=gen, device=dev)], 1)
    return torch.where(ground[:, None], flat, mu), (-2.5, 0.6), (0.5, 1.5)


def _morton(p):
    lo, hi = p.amin(0), p.amax(0)
    q = ((p - lo) / (hi - lo) * ((1 << 21) - 1)).long().clamp_(0, (1 << 21) - 1)
    code = torch.zeros(len(p), dtype=torch.int64, device=p.device)
    for x in range(3):
        v = q[:, x]
        for shift, mask in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F),
                            (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
            v = (v | (v << shift)) & mask
        code |= v << x
    return code


def _rotations(q):
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).view(*q.shape[:-1], 3, 3)


def _covariance(log_scale, quat):
    R = _rotations(quat)
    return ((R * (2 * log_scale).exp()[..., None, :])[..., None, :] * R[..., None, :, :]).sum(-1)


@lru_cache(maxsize=2)
def _scene(scene, leaves, degree):
    """A tree over Morton-ordered leaves: two to eight consecutive nodes to a parent, which is
    their weighted moment match along the axes.  Host arrays in the layout of ``synth.Tree``."""
    gen = torch.Generator(device="cuda").manual_seed(17 + leaves)
    mu, (ls_mean, ls_std), (op_mean, op_std) = _leaves(scene, leaves, gen)
    mu = mu[torch.sort(_morton(mu.double()), stable=True).indices]
    dev, K = mu.device, (degree + 1) ** 2
    normal = lambda *shape: torch.randn(*shape, generator=gen, device=dev)  # noqa: E731
    sh = normal(leaves, K, 3) * 0.05
    sh[:, 0] = (torch.rand(leaves, 3, generator=gen, device=dev) - 0.5) * (2.0 * math.sqrt(math.pi))
    levels = [dict(mu=mu, log_scale=ls_mean + ls_std * normal(leaves, 3), quat=normal(leaves, 4),
                   logit=op_mean + op_std * normal(leaves), sh=sh.view(leaves, -1))]
    sizes = []
    while len(levels[-1]["mu"]) > 1:
        c = levels[-1]
        n = len(c["mu"])
        ends = torch.randint(2, 9, (n // 2 + 1,), generator=gen, device=dev).cumsum(0)
        ends = torch.cat([ends[ends < n - 1], ends.new_tensor([n])])
        starts = torch.cat([ends.new_zeros(1), ends[:-1]])
        idx = starts[:, None] + torch.arange(9, device=dev)
        has = idx < ends[:, None]
        idx = idx.clamp(max=n - 1)
        w = (torch.sigmoid(c["logit"]) * c["log_scale"].sum(1).exp())[idx] * has
        w = w / w.sum(1, keepdim=True)
        m = (w[..., None] * c["mu"][idx]).sum(1)
        var = sum((w[:, k, None] * (_covariance(c["log_scale"][idx[:, k]], c["quat"][idx[:, k]]).diagonal(dim1=1, dim2=2)
                                    + (c["mu"][idx[:, k]] - m) ** 2)) for k in range(9))
        levels.append(dict(mu=m, log_scale=0.5 * var.clamp(min=1e-12).log(), quat=torch.eye(4, device=dev)[0].expand(len(m), 4),
                           logit=torch.where(has, c["logit"][idx], -math.inf).amax(1),
                           sh=sum(w[:, k, None] * c["sh"][idx[:, k]] for k in range(9))))
        sizes.append(ends - starts)
    levels, sizes = levels[::-1], sizes[::-1]
    counts = [len(x["mu"]) for x in levels]
    first = np.concatenate([[0], np.cumsum(counts)])
    n = int(first[-1])
    parent = torch.full((n,), -1, dtype=torch.int64, device=dev)
    for k in range(1, len(levels)):
        parent[first[k]:first[k + 1]] = first[k - 1] + torch.repeat_interleave(torch.arange(counts[k - 1], device=dev), sizes[k - 1])
    ap = torch.empty(len(levels) - 1, n, dtype=torch.int32, device=dev)
    a = parent
    for k in range(len(levels) - 1):
        ap[k] = a.to(torch.int32)                 # -1 past the root is the padding 0xFFFFFFFF
        a = torch.where(a >= 0, parent[a.clamp(min=0)], a)
    p = {k: torch.cat([x[k] for x in levels]) for k in levels[0]}
    cov = _covariance(p["log_scale"], p["quat"])
    opacity = torch.sigmoid(p["logit"].double())
    host = lambda t: t.contiguous().cpu().numpy()  # noqa: E731
    leaf = torch.zeros(n, dtype=torch.uint8, device=dev)
    leaf[first[-2]:] = 1
    level = np.repeat(np.arange(len(levels), dtype=np.int32), counts)
    return synth.Tree(mu=host(p["mu"].T), cov=host(torch.stack([cov[:, i, j] for i in range(3) for j in range(i, 3)])),
                      log_scale=host(p["log_scale"].T), quat=host(p["quat"].T), opacity=host(opacity.float()),
                      ln_opacity=host(opacity.log().float()), opacity_logit=host(p["logit"]), sh=host(p["sh"].view(n, K, 3)),
                      sh_degree=degree, parent=host(parent.to(torch.int32)), is_leaf=host(leaf), level=level,
                      ap=host(ap).view(np.uint32), name=scene)


def _camera(case, rng, width, height):
    """A pose of the scene's flight path."""
    a = rng.uniform(0, 2 * math.pi)
    if case["scene"] == "box":
        r = rng.uniform(60, 80)
        return synth.look_at_camera([r * math.cos(a), r * math.sin(a), 40.0], [0, 0, 0], width, height, 60.0)
    if case["scene"] == "blobs":
        return synth.look_at_camera([200 * math.cos(a), 200 * math.sin(a), 60.0], [0, 0, 25.0], width, height, 60.0)
    return synth.heading_pitch_camera([700 * math.cos(a), 700 * math.sin(a), rng.uniform(40, 60)], a + 0.5 * math.pi,
                                      rng.uniform(10, 20), width, height, 45.0)


def _cameras(case, seed):
    rng = np.random.default_rng(seed)
    cams = []
    for v in range(case["views"]):
        # a batch's viewers have windows of a third, two thirds, one and two of the case's size
        s = (1 / 3, 2 / 3, 1, 2)[v % 4] if case["kind"] == "batch" else 1
        cams.append(_camera(case, rng, max(1, int(case["width"] * s)), max(1, int(case["height"] * s))))
    return cams


def _params(case, seed):
    """The tree's parameters, moved a little, as after some training steps: float32, on the GPU."""
    t = _scene(case["scene"], case["leaves"], case["degree"])
    gen = torch.Generator(device="cuda").manual_seed(seed)
    p = dict(mu=t.mu, log_scale=t.log_scale, quat=t.quat, logit=t.opacity_logit, sh=t.sh)
    p = {k: torch.from_numpy(v).cuda() for k, v in p.items()}
    return {k: v + 0.01 * torch.randn(v.shape, generator=gen, device="cuda") for k, v in p.items()}


def _image(case, seed):
    """A target image (train) or an image gradient (accumulate), one for each view."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    shape = (case["views"], 3, case["height"], case["width"])
    return (torch.rand if case["kind"] == "train" else torch.randn)(*shape, generator=gen, device="cuda")


@lru_cache(maxsize=1)
def _program(scene, leaves, degree, tile, tau_R, tau, sizes):
    """What a program sets up once: the renderer with its tree and, for a batch, its windows and image buffers."""
    r = filtergs.Renderer(device=0, tau_R=tau_R, tile=tile, bg=(0.1, 0.2, 0.3))
    r.load_tree(_scene(scene, leaves, degree))
    r.shrink(*((tau, math.log(tau)) if tau else ()))
    images = None
    if sizes:
        r.batch_setup([synth.look_at_camera([0, -100, 50], [0, 0, 0], w, h, 60.0) for w, h in sizes])
        pixels = int(r.batch_offsets[-1])
        images = [torch.empty(k * pixels, device="cuda") for k in (3, 1)]
    return SimpleNamespace(r=r, images=images)


def prepare(case, seed):
    kind = case["kind"]
    cams = _cameras(case, seed)
    sizes = tuple((c.width, c.height) for c in cams) if kind == "batch" else ()
    keep = _program(case["scene"], case["leaves"], case["degree"], (case["tile_w"], case["tile_h"]), case["tau_R"], case["tau"], sizes)
    s = SimpleNamespace(kind=kind, cams=cams, r=keep.r, images=keep.images)
    if kind in ("train", "accumulate"):
        s.params, s.dL = _params(case, seed), _image(case, seed)
        if kind == "train":
            for v in s.params.values():
                v.requires_grad_()
        else:
            s.grads = {k: torch.empty_like(v) for k, v in s.params.items()}
    if kind == "serve":
        s.host = [torch.empty(k * case["height"] * case["width"], pin_memory=True).view(-1, case["height"], case["width"]) for k in (3, 1)]
        s.arrays = [x.numpy() for x in s.host]
    return s


def run(s):
    r = s.r
    if s.kind == "frame":
        r.set_camera(s.cams[0])
        rgb, T, _ = r.render()
        return {"rgb": rgb, "T": T}
    if s.kind == "serve":
        r.set_camera(s.cams[0])
        r.render_host(s.arrays[0], s.arrays[1], pipelined=True)
        return {"rgb": s.host[0], "T": s.host[1][0]}
    if s.kind == "batch":
        r.batch_set_cameras(s.cams)
        views = r.render_batch(*s.images, graph=True)[3]
        return {"views": [{"rgb": rgb, "T": T} for rgb, T in views]}
    if s.kind == "calibrate":
        out = []
        for cam in s.cams:
            r.set_camera(cam)
            gbar, G, _ = r.calibrate_view()
            out.append({"gbar": gbar, "G": G})
        return {"views": out}
    if s.kind == "train":
        for v in s.params.values():
            v.grad = None
        r.set_camera(s.cams[0])
        rgb = filtergs.render_differentiable(r, *(s.params[k] for k in PARAMS))
        (rgb - s.dL[0]).square().mean().backward()
        return {"rgb": rgb.detach(), **{k: s.params[k].grad for k in PARAMS}}
    r.update_params(s.params)
    images = []
    for v, cam in enumerate(s.cams):
        r.set_camera(cam)
        images.append(r.render()[0])
        r.backward(s.dL[v], s.params, s.grads, accumulate=v > 0)
    return {"rgb": images, **s.grads}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: the boxes of 128 nodes' centres, the visible nodes' centres, the selected nodes' attributes and SH,
    the images; for the differentiable form every parameter in, every gradient out.  Operations: 9 for each pixel and
    Gaussian tested and 24 for each that is blended, at the recipes' mean of 18 and 6 a pixel (three times both for
    the backward).  The selected share of a scene is the recipes'."""
    nodes = 1.25 * case["leaves"]
    rows = 3 * (case["degree"] + 1) ** 2
    pixels = sum(c.width * c.height for c in _cameras(case, 0))
    selected = {"box": 0.6, "blobs": 0.3, "city": 0.08}[case["scene"]] * nodes
    evaluations = pixels * (9 * 18 + 24 * 6)
    frame = nodes / 4 + selected * (12 + 48 + 4 * rows)
    if case["kind"] in ("train", "accumulate"):
        return {"bytes": nodes * 4 * (11 + rows) * 2 + case["views"] * frame + 24 * pixels, "flops": 4 * evaluations}
    image = 8 * pixels / 256 if case["kind"] == "calibrate" else 16 * pixels
    return {"bytes": (1 if case["kind"] == "batch" else case["views"]) * frame + image, "flops": evaluations}


# ---------------------------------------------------------------- the same in 64 bits
def exact(case, seed):
    cams = _cameras(case, seed)
    tree = _scene(case["scene"], case["leaves"], case["degree"])
    dev = torch.device("cuda")
    learning = case["kind"] in ("train", "accumulate")
    if learning:
        leaf = {k: v.double().requires_grad_() for k, v in _params(case, seed).items()}
        cov = _covariance(leaf["log_scale"].T, leaf["quat"].T)
        logit = leaf["logit"].clamp(-80, 80)
        g = dict(mu=leaf["mu"].T, cov=cov, opacity=torch.sigmoid(logit), ln_opacity=torch.nn.functional.logsigmoid(logit), sh=leaf["sh"])
    else:
        f64 = lambda x: torch.from_numpy(x).to(dev).double()  # noqa: E731
        c = f64(tree.cov)
        g = dict(mu=f64(tree.mu).T, cov=c[[0, 1, 2, 1, 3, 4, 2, 4, 5]].T.reshape(-1, 3, 3), opacity=f64(tree.opacity),
                 ln_opacity=f64(tree.ln_opacity), sh=torch.from_numpy(tree.sh).to(dev))
    images = _image(case, seed).double() if learning else None
    out, total = [], 0.0
    for v, cam in enumerate(cams):
        with torch.set_grad_enabled(learning):
            splat = _splats(case, tree, g, cam)
        pairs = _pairs(case, cam, splat)
        if case["kind"] == "calibrate":
            out.append(_blend(case, cam, splat, pairs, kpc=True))
            continue
        flat = {k: x.detach() for k, x in splat.items()}
        image = _blend(case, cam, flat, pairs)
        out.append({"rgb": image[0], "T": image[1]})
        if learning:
            dL = 2 * (image[0] - images[v]) / image[0].numel() if case["kind"] == "train" else images[v]
            keys = [k for k, x in splat.items() if x.requires_grad]
            rest = {k: flat[k].clone().requires_grad_() if k in keys else flat[k] for k in flat}
            _blend(case, cam, rest, pairs, dL=dL)
            torch.autograd.backward([splat[k] for k in keys], [torch.zeros_like(rest[k]) if rest[k].grad is None else rest[k].grad for k in keys],
                                    retain_graph=v + 1 < len(cams))
    if case["kind"] in ("frame", "serve"):
        return out[0]
    if learning:
        rgb = out[0]["rgb"] if case["kind"] == "train" else [o["rgb"] for o in out]
        return {"rgb": rgb, **{k: leaf[k].grad for k in PARAMS}}
    return {"views": out}


def _screen(cam, mu, cov):
    dev = mu.device
    W = torch.from_numpy(cam.R).to(dev).double()
    x, y, z = (mu @ W.T + torch.from_numpy(cam.t).to(dev).double()).unbind(1)
    lx, ly = 1.3 * cam.tan_half_x, 1.3 * cam.tan_half_y
    seen = (z > 0.2) & ((x / z).abs() <= lx) & ((y / z).abs() <= ly)
    zero = torch.zeros_like(x)
    J = torch.stack([cam.fx / z, zero, -cam.fx * x / z ** 2, zero, cam.fy / z, -cam.fy * y / z ** 2], 1).view(-1, 2, 3) @ W
    S = (J[:, :, :, None] * cov[:, None]).sum(2)
    S = (S[:, :, None] * J[:, None]).sum(3)
    a, b, c = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det, mid = a * c - b * b, 0.5 * (a + c)
    lam = mid + (mid * mid - det).clamp(min=0.1).sqrt()
    return SimpleNamespace(x=x, y=y, z=z, seen=seen, a=a, b=b, c=c, det=det, lam=lam)


def _splats(case, tree, g, cam):
    """The cut, projected: per selected Gaussian centre, conic, opacity, colour, depth and radius."""
    dev = g["mu"].device
    with torch.no_grad():
        s = _screen(cam, g["mu"], g["cov"])
        passes = s.seen & (torch.from_numpy(tree.is_leaf).to(dev).bool() | (3 * s.lam.sqrt() <= case["tau_R"]))
        parent = torch.from_numpy(tree.parent).to(dev).long()
        below = torch.zeros_like(passes)          # an ancestor passes
        first = np.concatenate([[0], np.cumsum(np.bincount(tree.level))])
        for a, b in zip(first[1:-1], first[2:]):
            p = parent[a:b]
            below[a:b] = below[p] | passes[p]
        sel = (passes & ~below).nonzero()[:, 0]
    mu = g["mu"][sel]
    s = _screen(cam, mu, g["cov"][sel])
    ln_a = g["ln_opacity"][sel]
    r = 3 * s.lam.sqrt()
    if case["tau"] and case["kind"] != "calibrate":       # calibration is done on the 3-sigma footprint
        q = 2 * (ln_a - float(np.float32(math.log(case["tau"]))))
        r = torch.where(q > 0, torch.minimum(r, (s.lam * q.clamp(min=0)).sqrt()), torch.full_like(r, -1.0))
    d = mu - torch.from_numpy(cam.campos).to(dev).double()
    d = d / d.norm(dim=1, keepdim=True)
    colour = (_harmonics(d, case["degree"])[:, :, None] * g["sh"][sel].double()).sum(1) + 0.5
    return dict(u=cam.fx * s.x / s.z + cam.cx, v=cam.fy * s.y / s.z + cam.cy, A=s.c / s.det, B=-s.b / s.det, C=s.a / s.det,
                opacity=g["opacity"][sel], rgb=colour.clamp(min=0), ln_a=ln_a.detach(), z=s.z.detach(), r=r.detach())


def _harmonics(d, degree):
    """Real spherical harmonics with the Condon-Shortley phase, from their Cartesian forms."""
    x, y, z = d.unbind(1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if degree > 0:
        n = math.sqrt(3 / (4 * pi))
        Y += [-n * y, n * z, -n * x]
    if degree > 1:
        n = 0.5 * math.sqrt(15 / pi)
        Y += [n * x * y, -n * y * z, 0.25 * math.sqrt(5 / pi) * (2 * z * z - x * x - y * y), -n * x * z, 0.5 * n * (x * x - y * y)]
    if degree > 2:
        a, b, c = 0.25 * math.sqrt(35 / (2 * pi)), 0.25 * math.sqrt(105 / pi), 0.25 * math.sqrt(21 / (2 * pi))
        Y += [-a * y * (3 * x * x - y * y), 2 * b * x * y * z, -c * y * (4 * z * z - x * x - y * y),
              0.25 * math.sqrt(7 / pi) * z * (2 * z * z - 3 * x * x - 3 * y * y), -c * x * (4 * z * z - x * x - y * y),
              b * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


@torch.no_grad()
def _pairs(case, cam, s):
    """(tile, Gaussian) of every pair, by tile, then depth, then rank; and each tile's first pair."""
    tw, th = case["tile_w"], case["tile_h"]
    tx, ty = -(-cam.width // tw), -(-cam.height // th)
    ok = (s["r"] >= 0) & (s["A"] > 0)
    x0, x1 = ((s["u"] - s["r"]) / tw).floor().clamp(0, tx), (((s["u"] + s["r"]) / tw).floor() + 1).clamp(0, tx)
    y0, y1 = ((s["v"] - s["r"]) / th).floor().clamp(0, ty), (((s["v"] + s["r"]) / th).floor() + 1).clamp(0, ty)
    w, h = (x1 - x0).clamp(min=0).long(), (y1 - y0).clamp(min=0).long()
    n = w * h * ok
    order = torch.sort(s["z"], stable=True).indices
    n = n[order]
    who = torch.repeat_interleave(order, n)
    k = torch.arange(len(who), device=n.device) - torch.repeat_interleave(n.cumsum(0) - n, n)
    tile = (y0[who].long() + k // w[who]) * tx + x0[who].long() + k % w[who]
    tile, order = torch.sort(tile, stable=True)
    first = torch.searchsorted(tile, torch.arange(tx * ty + 1, device=n.device))
    return who[order], first, tx


def _blend(case, cam, s, pairs, kpc=False, dL=None):
    """Eq. 2 tile by tile: the image and T; with kpc the tiles' GTC and their mean (Eq. 5-7); with dL the
    gradients are left in the splats' grad."""
    who, first, tx = pairs
    tw, th, dev = case["tile_w"], case["tile_h"], who.device
    counts = first[1:] - first[:-1]
    tiles = torch.sort(counts, stable=True).indices
    tiles = tiles[counts[tiles] > 0]
    lengths = counts[tiles].tolist()
    bg = torch.tensor([0.1, 0.2, 0.3], device=dev).double()
    ny = (len(first) - 1) // tx
    rgb = bg[:, None, None].expand(3, ny * th, tx * tw).clone()
    T_out = torch.ones(ny * th, tx * tw, dtype=torch.float64, device=dev)
    G = torch.full((len(first) - 1,), math.nan, dtype=torch.float64, device=dev)
    px = torch.arange(256, device=dev)
    cells = 8_000_000 if dL is not None else 24_000_000
    k = 0
    while k < len(lengths):
        e = k + 1
        while e < len(lengths) and (e + 1 - k) * lengths[e] * 256 <= cells:
            e += 1
        t, L = tiles[k:e], lengths[e - 1]
        k = e
        j = torch.arange(L, device=dev)
        has = j < counts[t][:, None]
        m = who[(first[t][:, None] + j).clamp(max=len(who) - 1)]
        x, y = (t % tx * tw)[:, None] + px % tw, (t // tx * th)[:, None] + px // tw
        inside = (x < cam.width) & (y < cam.height)
        dx, dy = s["u"][m][..., None] - (x + 0.5)[:, None], s["v"][m][..., None] - (y + 0.5)[:, None]
        power = -0.5 * (s["A"][m][..., None] * dx * dx + s["C"][m][..., None] * dy * dy) - s["B"][m][..., None] * dx * dy
        hit = has[..., None] & (power <= 0) & (power >= -math.log(255) - s["ln_a"][m][..., None])
        alpha = torch.where(hit, (s["opacity"][m][..., None] * power.clamp(max=0).exp()).clamp(max=0.99), 0.0)
        Tn = (1 - alpha).cumprod(1)
        on = Tn.detach() >= 1e-4
        weight = torch.where(on, alpha * torch.cat([torch.ones_like(Tn[:, :1]), Tn[:, :-1]], 1), 0.0)
        if kpc:
            G[t] = (weight * inside[:, None]).sum((1, 2)) / counts[t]
            continue
        last = on.sum(1)                                   # the Gaussians before the stop are a prefix
        T = torch.where(last > 0, Tn.gather(1, (last - 1).clamp(min=0)[:, None])[:, 0], 1.0)
        C = torch.einsum("blp,blc->cbp", weight, s["rgb"][m]) + bg[:, None, None] * T
        if dL is not None:
            at = dL[:, y.clamp(max=cam.height - 1), x.clamp(max=cam.width - 1)]
            torch.where(inside, C * at, 0.0).sum().backward()
        else:
            rgb[:, y, x], T_out[y, x] = C, T
    if kpc:
        used = ~G.isnan()
        return {"gbar": float(G[used].mean()) if used.any() else math.nan, "G": G}
    return rgb[:, :cam.height, :cam.width], T_out[:cam.height, :cam.width]
