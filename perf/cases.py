"""Performance cases of the differentiable Gaussian rasterizer.

The work a user has the library do: whole training steps (small to large,
one view or a batch of views of uneven size, captured in a CUDA graph or
eager through autograd), a forward-only render, and the single stages that a
program can call by themselves (projection, list construction, blending and
its adjoint, loss).

A case is a dict of plain values:
  kind    step | train | render | project | lists | blend | loss
  scene   box (means uniform in a box, as dense as its log-scales make it) or
          clusters (means from 64 anisotropic clusters, SH up to `degree`)
  n, degree, width, height, views, tile, attr (record staging), ls (mean
  log-scale), opacity (mean opacity logit), lam (weight of D-SSIM in the loss)
Scenes, cameras and targets are drawn on the GPU from the seed alone.
"""
import math

import numpy as np
import torch

from paper_2603_09277_gb300 import scenes
from paper_2603_09277_gb300.rasterize import (PARAM_KEYS, Rasterizer, capture_step,
                                              l1_entropy_loss, rasterize, sh_layout_for)

GAMMA = scenes.GAMMA
STRIDE = 16  # SH coefficients stored per Gaussian

_BASE = {"scene": "box", "n": 10_000, "degree": 0, "width": 256, "height": 256, "views": 1,
         "tile": 16, "attr": "f32", "ls": -3.5, "opacity": 0.0, "lam": 0.0}


def _case(kind, **kw):
    return {"kind": kind, **_BASE, **kw}


def listed():
    return [
        # a training step at the smallest scene (10k Gaussians, 256x256), replayed from a graph
        _case("step", name="step_10k_256"),
        # early training: an initial point cloud of 100k Gaussians, coarse resolution, SH degree 1
        _case("step", name="step_100k_sh1", scene="clusters", n=100_000, degree=1, width=618,
              height=411, ls=-3.5),
        # a training step at scene scale: 1M Gaussians, SH degree 3, one outdoor view
        _case("step", name="step_1M_sh3", scene="clusters", n=1_000_000, degree=3, width=1237,
              height=822, ls=-4.0),
        # the batched step: 3M Gaussians, 8 views of three sizes
        _case("step", name="step_3M_8views", n=3_000_000, width=1237, height=822, views=8),
        # mixed precision: 3M Gaussians, one 1080p view, BF16 records
        _case("step", name="step_3M_bf16_1080p", n=3_000_000, width=1920, height=1080,
              attr="bf16"),
        # an eager training iteration through autograd with D-SSIM, 8-px tiles
        _case("train", name="train_200k_tile8", scene="clusters", n=200_000, degree=2, width=641,
              height=427, tile=8, ls=-4.0, lam=0.2),
        # viewing a trained scene: projection, lists and blending of one 1080p view, eager
        _case("render", name="render_1M_1080p", scene="clusters", n=1_000_000, degree=3,
              width=1920, height=1080, ls=-4.0),
        # projection of a large scene with the 2D attributes that densification reads
        _case("project", name="project_1M_4views", scene="clusters", n=1_000_001, degree=3,
              width=979, height=546, views=4, ls=-4.0),
        # list construction alone: three views of a mid-size scene
        _case("lists", name="lists_400k_3views", n=400_000, width=979, height=546, views=3),
        # blending and its adjoint alone, large opaque splats (lists far longer than the walks)
        _case("blend", name="blend_30k_opaque", n=30_011, width=979, height=546, ls=-2.8,
              opacity=2.0),
        # the loss with D-SSIM on two views
        _case("loss", name="loss_dssim_2views", n=1, width=1237, height=822, views=2, lam=0.2),
    ]


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["step", "step", "step", "train", "render", "project", "lists", "blend",
                       "loss"])
    c = _case(kind, width=log_int(120, 1920))
    c["height"] = max(64, int(c["width"] * rng.uniform(0.5, 1.0)))
    c["views"] = rng.choice([1, 1, 2, 3, 5])
    if kind in ("train", "render"):
        c["views"] = 1
    if kind == "loss":
        c["n"] = 1
        c["lam"] = rng.choice([0.0, 0.2])
        return c
    c["scene"] = rng.choice(["box", "clusters"])
    if c["scene"] == "box":
        c["n"] = log_int(2_000, 600_000)
        # from the box's own density to sizes that shrink as the count grows
        c["ls"] = -3.5 + rng.choice([0.0, math.log((1e4 / max(c["n"], 10_000)) ** (1 / 3))])
        c["opacity"] = rng.choice([0.0, 2.0])
    else:
        c["n"] = log_int(5_000, 1_500_000)
        c["degree"] = rng.choice([0, 1, 2, 3])
        c["ls"] = rng.uniform(-4.5, -3.5)
    if kind == "lists":
        c["n"], c["views"] = min(c["n"], 400_000), min(c["views"], 3)
    c["tile"] = rng.choice([16, 16, 16, 8])
    c["attr"] = rng.choice(["f32", "f32", "f32", "bf16", "f16"])
    if kind == "train":
        c["lam"] = rng.choice([0.0, 0.2])
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _sizes(case):
    """View sizes: the first third at a quarter of width x height, the next at
    a half, the last at full size (one or two views: full size only)."""
    V, w, h = case["views"], case["width"], case["height"]
    if V < 3:
        return [(w, h)] * V
    return [(max(16, w >> (2 - 3 * v // V)), max(16, h >> (2 - 3 * v // V))) for v in range(V)]


def _cameras(case, seed):
    rng = np.random.default_rng(seed)
    sizes = _sizes(case)
    if case["scene"] == "box":
        yaws = [0.0] + list(rng.uniform(-15.0, 15.0, len(sizes) - 1))
        return scenes.yaw_cameras(sizes, yaws)
    cams = []
    for w, h in sizes:  # an orbit of radius 4 inside the ball, looking at its centre
        th = rng.uniform(0.0, 2.0 * math.pi)
        pos = np.array([4.0 * math.cos(th), 0.5, 4.0 * math.sin(th)])
        cams.append(scenes.camera(w, h, w, scenes.look_at(pos, (0.0, 0.0, 0.0)), pos))
    return cams


def _scene(case, seed):
    """Parameters on the GPU (the SH coefficients in the layout the degree takes)."""
    n, dev = case["n"], "cuda"
    g = torch.Generator(device=dev).manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device=dev)

    def uniform(*shape):
        return torch.rand(*shape, generator=g, device=dev)

    lay = sh_layout_for(case["degree"], STRIDE)
    K = (case["degree"] + 1) ** 2
    sh = torch.zeros((n, STRIDE, 3) if lay == 0 else (STRIDE, n, 3), device=dev)
    by_coef = sh.transpose(0, 1) if lay == 0 else sh
    if case["scene"] == "box":
        ar = min(1.0, case["height"] / case["width"])
        means = uniform(n, 3) * torch.tensor([2.0, 2.0 * ar, 4.0], device=dev) + torch.tensor(
            [-1.0, -ar, 2.0], device=dev)
        by_coef[0] = (uniform(n, 3) * 2.0 - 1.0) * math.sqrt(math.pi)
        ls_std = 0.5
    else:
        u = normal(64, 3)
        centres = u / u.norm(dim=1, keepdim=True) * 10.0 * uniform(64, 1) ** (1.0 / 3.0)
        w, x, y, z = torch.nn.functional.normalize(normal(64, 4)).unbind(1)
        rots = torch.stack([
            1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
            2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
            2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
        rots = rots * (uniform(64, 1, 3) * 1.7 + 0.3)  # axis standard deviations
        k = torch.randint(0, 64, (n,), generator=g, device=dev)
        means = centres[k] + torch.einsum("nij,nj->ni", rots[k], normal(n, 3))
        r = means.norm(dim=1, keepdim=True)
        means = means * torch.clamp(10.0 / r, max=1.0)
        by_coef[:K] = 0.2 * normal(K, n, 3)
        ls_std = 0.7
    q = normal(n, 4)
    return {"means": means.contiguous(), "log_scales": case["ls"] + ls_std * normal(n, 3),
            "quats": q / q.norm(dim=1, keepdim=True),
            "opacity_logits": case["opacity"] + normal(n), "sh": sh,
            "sh_degree": case["degree"], "sh_layout": lay}


def _targets(cams, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    return torch.rand(sum(c["width"] * c["height"] for c in cams), 3, generator=g, device="cuda")


def _inputs(case, seed):
    cams = _cameras(case, seed)
    return cams, _scene(case, seed), _targets(cams, seed), scenes.params(
        sh_degree=case["degree"], tile=case["tile"])


def _capacity(case):
    """Pairs a program reserves for the lists: 64 tiles of 16 px per row at a
    width of 1237 (the lists' own call returns the buffer whole)."""
    per_row = 64.0 * (16 / case["tile"]) ** 2 * (max(case["width"], 618) / 1237.0) ** 2
    return int(case["n"] * case["views"] * per_row)


def prepare(case, seed):
    cams, p, target, prm = _inputs(case, seed)
    kind = case["kind"]
    r = Rasterizer(cams, prm, case["n"], sh_stride=STRIDE, attr_dtype=case["attr"],
                   keep_debug=kind == "project",
                   pair_capacity=_capacity(case) if kind == "lists" else None)
    s = {"kind": kind, "r": r, "p": p, "target": target, "lam": case["lam"]}
    if kind == "step":
        # eager once (sizes the pair buffers), then captured as a training loop keeps it
        r.step(p, target, GAMMA)
        torch.cuda.synchronize()
        s["graph"] = capture_step(lambda: r.step(p, target, GAMMA, sync=False))
    elif kind == "train":
        for k in PARAM_KEYS:
            p[k].requires_grad_(True)
        r.preprocess(p)
        r.bin_sort()  # sizes the pair buffers
    elif kind == "project":
        # the rows of culled Gaussians are left as they are by the call
        for t in (r.mean2d, r.conic_opacity, r.rgb):
            t.zero_()
    elif kind == "loss":
        g = torch.Generator(device="cuda").manual_seed(seed + 2)
        # an image as far from its target as in training
        r.image.copy_((target + 0.1 * torch.randn(target.shape, generator=g, device="cuda"))
                      .clamp_(0.0, 1.0))
        r.entropy.copy_(2.0 * torch.rand(r.entropy.shape, generator=g, device="cuda"))
    else:
        r.preprocess(p)
        r.bin_sort()
        if kind == "lists":
            r.sorted_vals.zero_()
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(s):
    kind, r, p = s["kind"], s["r"], s["p"]
    if kind == "step":
        s["graph"].replay()
        return {"image": r.image, "entropy": r.entropy, "loss": r.loss_dev, "grads": dict(r.grads),
                "status": r.status_dev}
    if kind == "train":
        for k in PARAM_KEYS:
            p[k].grad = None
        image, entropy = rasterize(p, r)
        loss = l1_entropy_loss(image, entropy, s["target"], r, GAMMA, s["lam"])
        loss.backward()
        return {"image": image, "entropy": entropy, "loss": loss,
                "grads": {k: p[k].grad for k in PARAM_KEYS}}
    if kind == "render":
        r.preprocess(p)
        r.bin_sort()
        r.render_fwd()
        return {"image": r.image, "entropy": r.entropy, "T": r.final_T, "last": r.last_idx}
    if kind == "project":
        r.preprocess(p)
        return {"mean2d": r.mean2d, "conic_opacity": r.conic_opacity, "rgb": r.rgb,
                "depth": r.depth, "radius": r.radius, "tiles_touched": r.tiles_touched}
    if kind == "lists":
        r.bin_sort(sync=False)
        return {"vals": r.sorted_vals, "ranges": r.tile_ranges, "pairs": r.num_pairs_dev}
    if kind == "blend":
        r.render_fwd()
        r.loss(s["target"], GAMMA)
        r.render_bwd(p)
        return {"image": r.image, "entropy": r.entropy, "loss": r.loss_dev, "grads": dict(r.grads)}
    r.loss(s["target"], GAMMA, lam=s["lam"])
    return {"loss": r.loss_dev, "dL_dimage": r.dL_dimage, "dL_dentropy": r.dL_dentropy}


def work(case):
    """Bytes: each input read once, each output written once.  Operations:
    the projection (about 250 per row) and its adjoint (about 500)."""
    kind, n, V = case["kind"], case["n"], case["views"]
    px = sum(w * h for w, h in _sizes(case))
    K = (case["degree"] + 1) ** 2
    params, grads = n * (44 + 12 * K), n * (44 + 12 * STRIDE)
    if kind in ("step", "train"):
        return {"bytes": params + grads + px * (12 + 16), "flops": 750.0 * n * V}
    if kind == "render":
        return {"bytes": params + px * 24, "flops": 250.0 * n * V}
    if kind == "project":
        return {"bytes": params + n * V * 48, "flops": 250.0 * n * V}
    if kind == "lists":
        pairs = 0
        for c in _cameras(case, 0):
            q = _project64(_scene64(case, _scene(case, 0)), c, case["tile"])
            pairs += int(((q["x1"] - q["x0"]) * (q["y1"] - q["y0"])).sum())
        return {"bytes": n * V * 16 + 4 * pairs, "flops": 0.0}
    if kind == "blend":
        return {"bytes": params + grads + px * (12 + 16), "flops": 500.0 * n * V}
    return {"bytes": px * (12 + 12 + 4 + 12 + 4), "flops": px * 3.0 * (640 if case["lam"] else 4)}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits, from the definitions, in plain torch
# ---------------------------------------------------------------------------
#: Pixel tests per view above which the 64-bit pass would take over about 20 seconds.
_MOST_TESTS = 3_000_000_000


def _sh_basis(d):
    x, y, z = d.unbind(1)
    xx, yy, zz = x * x, y * y, z * z
    pi = math.pi
    a, b, c = (math.sqrt(k / pi) for k in (15.0, 5.0, 15.0))
    e, f, g, h = (math.sqrt(k / pi) for k in (35.0 / 2, 105.0, 21.0 / 2, 7.0))
    s1 = math.sqrt(3.0 / (4 * pi))
    return torch.stack([
        torch.full_like(x, 0.5 / math.sqrt(pi)), -s1 * y, s1 * z, -s1 * x,
        a / 2 * x * y, -a / 2 * y * z, b / 4 * (2 * zz - xx - yy), -a / 2 * x * z,
        c / 4 * (xx - yy), -e / 4 * y * (3 * xx - yy), f / 2 * x * y * z,
        -g / 4 * y * (4 * zz - xx - yy), h / 4 * z * (2 * zz - 3 * xx - 3 * yy),
        -g / 4 * x * (4 * zz - xx - yy), f / 4 * z * (xx - yy), -e / 4 * x * (xx - 3 * yy)], 1)


def _scene64(case, p):
    q = {k: p[k].detach().double() for k in PARAM_KEYS}
    if p["sh_layout"] == 1:
        q["sh"] = q["sh"].transpose(0, 1).contiguous()
    q["degree"] = case["degree"]
    return q


def _project64(p, cam, tile):
    """EWA projection of every Gaussian into one view; differentiable."""
    prm = {k: float(np.float32(v)) for k, v in scenes.DEFAULT_PARAMS.items()}
    dev = p["means"].device
    M = torch.tensor(np.asarray(cam["world_to_cam"]), dtype=torch.float64, device=dev)
    R, t = M[:, :3], M[:, 3]
    W, H, fx, fy = cam["width"], cam["height"], cam["fx"], cam["fy"]
    m = p["means"]
    zr = ((R[2, 0] * m[:, 0] + R[2, 1] * m[:, 1]) + R[2, 2] * m[:, 2]) + t[2]
    depth = zr.detach().float()
    vis = depth > prm["near_z"]
    tc = m @ R.T + t
    z = torch.where(vis, tc[:, 2], torch.ones_like(zr))
    ux, uy = tc[:, 0] / z, tc[:, 1] / z
    lx, ly = prm["fov_clamp"] * 0.5 * W / fx, prm["fov_clamp"] * 0.5 * H / fy
    cux, cuy = ux.clamp(-lx, lx), uy.clamp(-ly, ly)
    o = torch.zeros_like(z)
    J = torch.stack([torch.stack([fx / z, o, -fx * cux / z], 1),
                     torch.stack([o, fy / z, -fy * cuy / z], 1)], 1)
    q = p["quats"] / p["quats"].norm(dim=1, keepdim=True)
    w, x, y, k = q.unbind(1)
    Rq = torch.stack([
        1 - 2 * (y * y + k * k), 2 * (x * y - w * k), 2 * (x * k + w * y),
        2 * (x * y + w * k), 1 - 2 * (x * x + k * k), 2 * (y * k - w * x),
        2 * (x * k - w * y), 2 * (y * k + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    N = (J @ R) @ (Rq * torch.exp(p["log_scales"])[:, None, :])
    S = N @ N.transpose(1, 2)
    A, B, C = S[:, 0, 0] + prm["dilation"], S[:, 0, 1], S[:, 1, 1] + prm["dilation"]
    det = A * C - B * B
    mx, my = fx * ux + cam["cx"], fy * uy + cam["cy"]
    with torch.no_grad():
        lam = 0.5 * (A + C) + torch.sqrt((0.5 * (A - C)) ** 2 + B * B)
        r = torch.ceil(3.0 * torch.sqrt(lam))
        TX, TY = -(-W // tile), -(-H // tile)
        x0 = ((mx - r) / tile).floor().clamp(0, TX).long()
        x1 = (((mx + r) / tile).floor() + 1).clamp(0, TX).long()
        y0 = ((my - r) / tile).floor().clamp(0, TY).long()
        y1 = (((my + r) / tile).floor() + 1).clamp(0, TY).long()
        vis = vis & (x1 > x0) & (y1 > y0)
        x1, y1 = torch.where(vis, x1, x0), torch.where(vis, y1, y0)
    cp = torch.tensor(np.asarray(cam["cam_pos"]), dtype=torch.float64, device=dev)
    d = m - cp
    K = (p["degree"] + 1) ** 2
    Y = _sh_basis(d / d.norm(dim=1, keepdim=True))[:, :K]
    rgb = torch.clamp((Y[:, :, None] * p["sh"][:, :K]).sum(1) + 0.5, min=0.0)
    a2d = torch.cat([torch.stack([mx, my, C / det, -B / det, A / det,
                                  torch.sigmoid(p["opacity_logits"])], 1), rgb], 1)
    return {"a2d": a2d, "depth": depth, "vis": vis, "x0": x0, "x1": x1, "y0": y0, "y1": y1,
            "TX": TX, "TY": TY}


def _lists64(q):
    """Gaussian ids per tile by (tile, FP32 depth, id), and the lists' starts and lengths."""
    g = torch.nonzero(q["vis"])[:, 0]
    g = g[torch.argsort(q["depth"][g], stable=True)]
    w = q["x1"][g] - q["x0"][g]
    area = w * (q["y1"][g] - q["y0"][g])
    k = torch.repeat_interleave(torch.arange(g.numel(), device=g.device), area)
    at = torch.arange(k.numel(), device=g.device) - (torch.cumsum(area, 0) - area)[k]
    tile = (q["y0"][g][k] + at // w[k]) * q["TX"] + q["x0"][g][k] + at % w[k]
    order = torch.argsort(tile, stable=True)
    cnt = torch.bincount(tile, minlength=q["TX"] * q["TY"])
    return g[k[order]], torch.cumsum(cnt, 0) - cnt, cnt


def _blend64(a2d, ids, ok, px):
    """Colour, T and entropy of tiles [G] of pixels px [G, S, 2] over their lists ids [G, L]."""
    prm = {k: float(np.float32(v)) for k, v in scenes.DEFAULT_PARAMS.items()}
    a = a2d[ids]
    dx = px[:, None, :, 0] - a[:, :, 0, None]
    dy = px[:, None, :, 1] - a[:, :, 1, None]
    e = -0.5 * (a[:, :, 2, None] * dx * dx + 2 * a[:, :, 3, None] * dx * dy
                + a[:, :, 4, None] * dy * dy)
    al = torch.clamp(a[:, :, 5, None] * torch.exp(e), max=prm["alpha_max"])
    al = torch.where((al.detach() >= prm["alpha_min"]) & ok[:, :, None], al, torch.zeros_like(al))
    with torch.no_grad():
        keep = torch.cumprod(1 - al, 1) >= prm["t_min"]
    al = torch.where(keep, al, torch.zeros_like(al))
    lt = torch.cumsum(torch.log1p(-al), 1)
    T = torch.exp(lt[:, -1])
    w = al * torch.exp(torch.cat([torch.zeros_like(lt[:, :1]), lt[:, :-1]], 1))
    on = w.detach() > 0
    h = -(w * torch.log(torch.where(on, w, torch.ones_like(w)))).sum(1) - T * torch.log(T)
    return torch.einsum("gls,glc->gsc", w, a[:, :, 6:9]), T, h


def _tiles64(q, lists, cam, tile, a2d, f):
    """Calls f(pixel ids [G, S], inside [G, S], colour, T, H) for groups of tiles."""
    ids, start, cnt = lists
    dev, W, H = ids.device, cam["width"], cam["height"]
    j = torch.arange(tile, device=dev)
    order = torch.argsort(cnt, descending=True)
    lens = cnt[order].tolist()
    i = 0
    while i < len(lens):
        L = max(lens[i], 1)
        G = max(1, min(len(lens) - i, 12_000_000 // (L * tile * tile)))
        t = order[i:i + G]
        i += G
        x = ((t % q["TX"]) * tile)[:, None, None] + j[None, None, :]
        y = ((t // q["TX"]) * tile)[:, None, None] + j[None, :, None]
        x, y = (v.expand(len(t), tile, tile).reshape(len(t), -1) for v in (x, y))
        at = start[t][:, None] + torch.arange(L, device=dev)
        ok = torch.arange(L, device=dev) < cnt[t][:, None]
        px = torch.stack([x, y], 2).double() + 0.5
        k = ids[torch.where(ok, at, 0)] if ids.numel() else torch.zeros_like(at)
        f(y * W + x, (x < W) & (y < H), *_blend64(a2d, k, ok, px))


def _loss64(image, target, entropy, cams, lam):
    total, off = 0.0, 0
    win = torch.exp(-0.5 * ((torch.arange(11, device=image.device).double() - 5) / 1.5) ** 2)
    win = win / win.sum()
    lam = float(np.float32(lam))
    gamma = float(np.float32(GAMMA))
    for c in cams:
        W, H = c["width"], c["height"]
        a, b = image[off:off + W * H], target[off:off + W * H]
        l1 = (a - b).abs().mean()
        v = (1 - lam) * l1 + gamma * entropy[off:off + W * H].mean()
        if lam > 0:
            x, y = (k.view(H, W, 3).permute(2, 0, 1)[:, None] for k in (a, b))

            def blur(k):
                k = torch.nn.functional.conv2d(k, win.view(1, 1, 1, 11), padding=(0, 5))
                return torch.nn.functional.conv2d(k, win.view(1, 1, 11, 1), padding=(5, 0))

            mx, my = blur(x), blur(y)
            sx, sy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
            s = ((2 * mx * my + 1e-4) * (2 * sxy + 9e-4)
                 / ((mx * mx + my * my + 1e-4) * (sx + sy + 9e-4)))
            v = v + lam * (1 - s.mean())
        total = total + v / len(cams)
        off += W * H
    return total


def exact(case, seed):
    cams, p, target, _ = _inputs(case, seed)
    kind, tile = case["kind"], case["tile"]
    target = target.double()
    if kind == "lists":
        return None  # whole numbers alone
    if kind == "loss":
        s = prepare(case, seed)["r"]
        img, ent = (t.double().requires_grad_(True) for t in (s.image, s.entropy))
        loss = _loss64(img, target, ent, cams, case["lam"])
        loss.backward()
        return {"loss": loss.detach().reshape(1), "dL_dimage": img.grad, "dL_dentropy": ent.grad}
    q64 = _scene64(case, p)
    if kind == "project":
        a, d = [], []
        for c in cams:
            q = _project64(q64, c, tile)
            a.append(torch.where(q["vis"][:, None], q["a2d"], torch.zeros_like(q["a2d"])))
            d.append(q["depth"].double())
        a = torch.cat(a)
        return {"mean2d": a[:, 0:2], "conic_opacity": a[:, 2:6], "rgb": a[:, 6:9],
                "depth": torch.cat(d), "radius": None, "tiles_touched": None}
    leaves = [q64[k].requires_grad_(True) for k in PARAM_KEYS]
    views = []
    for c in cams:
        with torch.no_grad():
            q = _project64(q64, c, tile)
            pairs = int(((q["x1"] - q["x0"]) * (q["y1"] - q["y0"])).sum())
        if pairs * tile * tile > _MOST_TESTS:
            return None
        views.append((q, _lists64(q)))
    img = torch.zeros_like(target)
    T, ent = torch.ones_like(target[:, 0]), torch.zeros_like(target[:, 0])
    off = 0
    with torch.no_grad():
        for c, (q, lists) in zip(cams, views):
            def put(pix, inside, col, t, h, off=off):
                at = (off + pix)[inside]
                img[at], T[at], ent[at] = col[inside], t[inside], h[inside]

            _tiles64(q, lists, c, tile, q["a2d"], put)
            off += c["width"] * c["height"]
    if kind == "render":
        return {"image": img, "entropy": ent, "T": T, "last": None}
    im, en = img.clone().requires_grad_(True), ent.clone().requires_grad_(True)
    loss = _loss64(im, target, en, cams, case["lam"])
    loss.backward()
    off = 0
    for c, (q, lists) in zip(cams, views):
        a2d = q["a2d"].detach().requires_grad_(True)

        def back(pix, inside, col, t, h, off=off):
            at = (off + pix)[inside]
            torch.autograd.backward([col[inside], h[inside]], [im.grad[at], en.grad[at]])

        _tiles64(q, lists, c, tile, a2d, back)
        out = _project64(q64, c, tile)["a2d"]
        touched = a2d.grad.abs().sum(1) > 0  # (rows behind the camera hold no value)
        out[touched].backward(a2d.grad[touched])
        off += c["width"] * c["height"]
    grads = {k: t.grad for k, t in zip(PARAM_KEYS, leaves)}
    if p["sh_layout"] == 1:
        grads["sh"] = grads["sh"].transpose(0, 1)
    if case["attr"] != "f32":  # (16-bit records: the gradients are those of rounded inputs)
        grads = dict.fromkeys(grads)
    loss = loss.detach()
    out = {"image": img, "entropy": ent, "grads": grads,
           "loss": loss if kind == "train" else loss.reshape(1)}
    return out if kind != "step" else {**out, "status": None}
