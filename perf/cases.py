"""What a user of this framework has it do, as cases that can be timed.

A case is one call sequence through the package's public entry points, over
the range of scenes and cameras that the workloads of ``synth`` and the
benchmark cover: 4 thousand to 2 million Gaussians, 1 to 64 cameras, 128 x 128
to 1920 x 1080 pixels, SH degrees 0 to 3.

``kind`` says which calls:

* ``train``    one training step: ``Renderer.step`` with targets (forward, L1
               loss, backward to every parameter)
* ``infer``    one frame of a fixed scene: ``Renderer.step`` without targets on
               a forward-only plan, with the cached slice state
* ``autograd`` the differentiable render under a loss of the caller's own:
               ``render`` and its backward with a given dL/dC
* ``cache``    ``condition_cache``, run once for each new scene before inference
* ``axes``     ``scale_rotation``, the input of densification

Scenes follow the recipes of ``synth`` (same distributions, drawn on the GPU).
"""

from __future__ import annotations

import math

import torch

import paper_2410_04974_gb300 as sx

PARAMS = ("mu_p", "mu_d", "l_raw", "opacity_logit", "sh")
MIXED_SIZES = ((256, 256), (512, 384), (800, 800), (1024, 768))
LAMBDA = 0.35
BG = (1.0, 1.0, 1.0)


def _case(kind, scene, n, views, width, height, degree=3, tile_h=16, learn_lambda=False, store_aux=False, mixed=False):
    return {"kind": kind, "scene": scene, "n": n, "views": views, "width": width, "height": height, "degree": degree,
            "tile_h": tile_h, "learn_lambda": learn_lambda, "store_aux": store_aux, "mixed": mixed}


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # the smallest training step of the repository: few tiles, latency counts
        named("train_4k_128sq", "train", "cube", 4096, 1, 128, 128),
        # the headline training step
        named("train_300k_8x800sq", "train", "shell", 300_000, 8, 800, 800),
        # a large batch of views of four sizes
        named("train_500k_64mixed", "train", "shell", 500_000, 64, 0, 0, mixed=True),
        # the largest scene, strongly view dependent, full-HD views
        named("train_2M_4x1080p", "train", "view", 2_000_000, 4, 1920, 1080),
        # a caller's own loss on one view, as a plain training loop does
        named("autograd_200k_800sq", "autograd", "shell", 200_000, 1, 800, 800),
        # ragged images, an odd number of Gaussians, a lower SH degree, a learnable lambda_opa and stored walk lengths
        named("autograd_50k_ragged", "autograd", "shell", 50_003, 3, 613, 347, degree=1, tile_h=8, learn_lambda=True,
              store_aux=True),
        # viewing a small volumetric scene: one frame, launches count
        named("infer_vol6k_1408sq", "infer", "volume", 6_660, 1, 1408, 1408),
        # viewing a surface scene
        named("infer_surf175k_1408sq", "infer", "shell", 174_746, 1, 1408, 1408),
        # the test views of a volumetric scene, rendered in one batch
        named("infer_vol183k_20x1024sq", "infer", "volume", 182_981, 20, 1024, 1024),
        # preparing a scene for inference
        named("cache_183k", "cache", "volume", 182_981, 0, 0, 0),
        # the per-Gaussian axes that densification asks for
        named("axes_500k", "axes", "shell", 500_000, 0, 0, 0),
    ]


def draw(rng):
    """Another case of the same ranges."""
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("train", "train", "train", "infer", "infer", "infer", "autograd", "autograd", "cache", "axes"))
    if kind in ("cache", "axes"):
        return _case(kind, rng.choice(("shell", "volume", "view")), spread(5_000, 2_000_000), 0, 0, 0)
    scene = rng.choice(("cube", "shell", "shell", "volume", "view"))
    n = spread(4_000, 16_000 if scene == "cube" else 600_000)
    views = 1 if kind == "infer" and rng.random() < 0.6 else spread(1, 16)
    width = spread(96, 1920)
    height = max(64, min(1408, int(width * rng.uniform(0.5, 1.1))))
    while views > 1 and views * width * height > 12_000_000:
        views -= 1
    return _case(kind, scene, n, views, width, height, degree=rng.choice((3, 3, 3, 2, 1, 0)),
                 tile_h=rng.choice((16, 16, 8)), learn_lambda=rng.random() < 0.25,
                 store_aux=kind == "autograd" and rng.random() < 0.5, mixed=kind != "infer" and rng.random() < 0.2)


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
class Camera:
    """A pinhole camera: x right, y down, z forward."""

    def __init__(self, pos, width, height, fov_x_deg=50.0):
        sub = [-p for p in pos]
        f = _unit(sub)
        right = _unit(_cross(f, (0.0, 1.0, 0.0) if abs(f[2]) > 0.999 else (0.0, 0.0, 1.0)))
        rows = (right, _cross(f, right), f)
        self.width, self.height, self.campos, self.znear = width, height, tuple(pos), 0.2
        self.fx = self.fy = (width / 2.0) / math.tan(math.radians(fov_x_deg) / 2.0)
        self.cx, self.cy = width / 2.0, height / 2.0
        self.world_to_cam = [[*r, -sum(a * b for a, b in zip(r, pos))] for r in rows]


def _cross(a, b):
    return (a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0])


def _unit(v):
    s = math.sqrt(sum(x * x for x in v))
    return tuple(x / s for x in v)


def _sizes(case):
    if case["mixed"]:
        return [MIXED_SIZES[(7 * k + k // 3) % 4] for k in range(case["views"])]
    return [(case["width"], case["height"])] * case["views"]


def _cameras(case):
    """Views on a ring (training) or spread over the upper hemisphere, at radius 4."""
    cams, v = [], case["views"]
    for k, (w, h) in enumerate(_sizes(case)):
        if case["kind"] != "infer" and not case["mixed"]:
            a = 2.0 * math.pi * k / v
            pos = (4.0 * math.cos(a), 4.0 * math.sin(a), 0.0)
        else:
            z = 0.087 + 0.913 * (k + 0.5) / v
            a = math.pi * (3.0 - math.sqrt(5.0)) * k
            r = math.sqrt(1.0 - z * z)
            pos = (4.0 * r * math.cos(a), 4.0 * r * math.sin(a), 4.0 * z)
        cams.append(Camera(pos, w, h))
    return cams


def _scene(case, seed):
    """Raw parameter planes of a scene, float32 on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, kind = case["n"], case["scene"]

    def normal(mean, std, *shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32) * std + mean

    def unit(m):
        v = normal(0.0, 1.0, 3, m)
        return v / v.norm(dim=0, keepdim=True)

    def uniform(lo, hi, *shape):
        return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float32) * (hi - lo) + lo

    pos, dp, logit = 0.01, 0.1, 0.0
    if kind == "cube":
        mu_p, pos, pos_off, dp = uniform(-1.0, 1.0, 3, n), 0.05, 0.02, 0.02
    elif kind == "volume":
        mu_p = normal(0.0, 0.6 / 1.7, 3, n)
        mu_p = mu_p / mu_p.norm(dim=0, keepdim=True).clamp(min=1.0)
        spacing = (4.0 / 3.0 * math.pi * 0.6 ** 3 / n) ** (1.0 / 3.0)
        pos, pos_off, dp, logit = 0.8 * spacing, 0.3 * spacing, 0.02, -1.0
    else:
        mu_p = unit(n) * normal(1.0, 0.01, 1, n)
        pos_off = 0.002 if kind == "view" else 0.004
    diag = torch.cat([normal(math.log(pos), 0.3, 3, n), normal(math.log(0.3), 0.3, 3, n)])
    off = torch.empty(15, n, device="cuda")
    off[:3] = normal(0.0, pos_off, 3, n)
    rows = ((3, 4, 5), (6, 7, 8), (10, 11, 12))     # direction-position entries of rows 3, 4, 5
    for j, r in enumerate(rows):
        if kind == "view":                          # direction strongly correlated with position
            c = unit(n) * uniform(0.0, 0.8, 1, n)
            off[list(r)] = 0.15 * c
            diag[3 + j] = torch.log(0.15 * torch.sqrt(1.0 - (c * c).sum(0)))
        else:
            off[list(r)] = normal(0.0, dp, 3, n)
    off[[9, 13, 14]] = 0.0 if kind == "view" else normal(0.0, 0.02, 3, n)
    p = {"mu_p": mu_p, "mu_d": unit(n), "l_raw": torch.cat([diag, 2.0 * torch.atanh(off.clamp(-0.99, 0.99))]),
         "opacity_logit": normal(logit, 1.0, n), "sh": normal(0.0, 0.2, (case["degree"] + 1) ** 2 * 3, n)}
    if case["learn_lambda"]:
        p["lambda_raw"] = normal(-0.619, 0.5, n)
    return {k: v.contiguous() for k, v in p.items()}


def _images(case, seed, photo):
    """Packed images of every view: smooth photo-like targets, or seeded dL/dC."""
    g = torch.Generator(device="cuda").manual_seed(seed + 77_777)
    out, total = [], 3 * sum(w * h for w, h in _sizes(case))
    for w, h in _sizes(case):
        if photo:
            small = torch.rand(1, 3, 12, 12, generator=g, device="cuda")
            img = torch.nn.functional.interpolate(small, size=(h, w), mode="bilinear", align_corners=False)[0]
            img = img + 0.02 * torch.randn(3, h, w, generator=g, device="cuda")
        else:
            img = torch.randn(3, h, w, generator=g, device="cuda") / total
        out.append(img.reshape(-1))
    return torch.cat(out)


def prepare(case, seed):
    s = {"kind": case["kind"], "params": _scene(case, seed)}
    if case["kind"] in ("cache", "axes"):
        return s
    p, train = s["params"], case["kind"] == "train"
    s["renderer"] = r = sx.Renderer(case["n"], case["degree"], _cameras(case), tile=(16, case["tile_h"]), lambda_opa=LAMBDA,
                                    bg=BG, store_aux=case["store_aux"], inference=case["kind"] == "infer")
    if case["kind"] == "infer":
        p["cond_cache"] = sx.condition_cache(p)
    r.forward(p)                                    # sizes the duplicate buffer
    s["images"] = r.new_images()
    if train:
        s["targets"] = _images(case, seed, True)
        s["grads"] = r.new_grads(p)
    elif case["kind"] == "autograd":
        s["grad_images"] = _images(case, seed, False)
        for t in p.values():
            t.requires_grad_()
    return s


def run(s):
    p = s["params"]
    if s["kind"] == "cache":
        return sx.condition_cache(p)
    if s["kind"] == "axes":
        rotation, scale, _ = sx.scale_rotation(p["l_raw"])
        return {"rotation": rotation, "scale": scale}
    r = s["renderer"]
    if s["kind"] == "infer":
        r.step(p, s["images"])
        return s["images"]
    if s["kind"] == "train":
        r.step(p, s["images"], s["targets"], grads=s["grads"])
        return {"images": s["images"], "loss": r.loss, "grads": s["grads"]}
    images = sx.render(r, p)
    grads = torch.autograd.grad(images, list(p.values()), s["grad_images"])
    return {"images": images, "grads": dict(zip(p, grads))}


def work(case):
    """Bytes: every parameter (or cached) plane and target read once, every image and gradient written once.  Operations:
    about 400 for the slice, colour and projection of one Gaussian in one view (three times that with its reverse), and 20 (90
    with the reverse) for each Gaussian that a pixel composites, of which these scenes have about 15 in a pixel."""
    n, k = case["n"], (case["degree"] + 1) ** 2 * 3
    if case["kind"] == "cache":
        return {"bytes": 4 * n * (22 + 25), "flops": 300 * n}
    if case["kind"] == "axes":
        return {"bytes": 4 * n * (21 + 12), "flops": 900 * n}
    pixels = sum(w * h for w, h in _sizes(case))
    lam = 1 if case["learn_lambda"] else 0
    if case["kind"] == "infer":
        return {"bytes": 4 * n * (6 + 25 + lam + k) + 12 * pixels, "flops": 400 * n * case["views"] + 20 * 15 * pixels}
    return {"bytes": 8 * n * (28 + lam + k) + 24 * pixels, "flops": 1200 * n * case["views"] + 90 * 15 * pixels}


# --------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# --------------------------------------------------------------------------
def _slice_state(p):
    """A = Spd Sd^-1, Sd^-1, Scond and alpha, with L = exp on the diagonal and tanh(raw / 2) below it."""
    n = p["l_raw"].shape[1]
    L = torch.zeros(n, 6, 6, dtype=torch.float64, device=p["l_raw"].device)
    i6 = torch.arange(6)
    L[:, i6, i6] = torch.exp(p["l_raw"][:6]).T
    low = torch.tril_indices(6, 6, -1)
    L[:, low[0], low[1]] = torch.tanh(0.5 * p["l_raw"][6:]).T
    S = L @ L.transpose(1, 2)
    Sp, Spd, Sd = S[:, :3, :3], S[:, :3, 3:], S[:, 3:, 3:]
    Sdi = torch.linalg.inv(Sd)
    A = Spd @ Sdi
    return A, Sdi, Sp - A @ Spd.transpose(1, 2)


def _sh(deg, d):
    x, y, z = d
    xx, yy, zz = x * x, y * y, z * z
    pi = math.pi
    c = lambda a, b: math.sqrt(a / (b * pi))  # noqa: E731
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if deg > 0:
        Y += [c(3, 4) * y, c(3, 4) * z, c(3, 4) * x]
    if deg > 1:
        Y += [c(15, 4) * x * y, c(15, 4) * y * z, c(5, 16) * (3 * zz - 1), c(15, 4) * x * z, c(15, 16) * (xx - yy)]
    if deg > 2:
        Y += [c(35, 32) * y * (3 * xx - yy), c(105, 4) * x * y * z, c(21, 32) * y * (5 * zz - 1),
              c(7, 16) * z * (5 * zz - 3), c(21, 32) * x * (5 * zz - 1), c(105, 16) * z * (xx - yy),
              c(35, 32) * x * (xx - 3 * yy)]
    return torch.stack(Y)


def _records(p, cond, cam, degree):
    """(u, v, conic a b c, alpha, r, g, b) of every Gaussian in one view, its depth, and its 2D variances."""
    A, Sdi, Sc = cond
    dev = p["mu_p"].device
    pos = torch.tensor(cam.campos, dtype=torch.float32, device=dev).double()
    w2c = torch.tensor(cam.world_to_cam, dtype=torch.float32, device=dev).double()
    fx, fy, cx, cy = (float(torch.tensor(v, dtype=torch.float32)) for v in (cam.fx, cam.fy, cam.cx, cam.cy))
    d = p["mu_p"] - pos[:, None]
    d = d / d.norm(dim=0, keepdim=True)
    delta = (d - p["mu_d"]).T
    lam = torch.sigmoid(p["lambda_raw"]) if "lambda_raw" in p else float(torch.tensor(LAMBDA, dtype=torch.float32))
    D = torch.einsum("ni,nij,nj->n", delta, Sdi, delta)
    alpha = torch.sigmoid(p["opacity_logit"]) * torch.exp(-lam * D)
    mc = p["mu_p"].T + torch.einsum("nij,nj->ni", A, delta)
    t = mc @ w2c[:, :3].T + w2c[:, 3]
    x, y, z = t.unbind(1)
    limx, limy = 1.3 * 0.5 * cam.width / fx, 1.3 * 0.5 * cam.height / fy
    rx, ry = (x / z).clamp(-limx, limx), (y / z).clamp(-limy, limy)
    o = torch.zeros_like(z)
    J = torch.stack([torch.stack([fx / z, o, -fx * rx / z], 1), torch.stack([o, fy / z, -fy * ry / z], 1)], 1)
    T = J @ w2c[:, :3]
    S2 = T @ Sc @ T.transpose(1, 2)
    a, b, c = S2[:, 0, 0] + 0.3, S2[:, 0, 1], S2[:, 1, 1] + 0.3
    det = a * c - b * b
    rgb = torch.sigmoid(torch.einsum("kn,kcn->cn", _sh(degree, d), p["sh"].view(-1, 3, p["sh"].shape[1])))
    rec = torch.stack([fx * x / z + cx, fy * y / z + cy, c / det, -b / det, a / det, alpha, *rgb], 1)
    return rec, z, (a.detach(), b.detach(), c.detach())


def _tile_lists(rec, z, var, cam, tw, th):
    """Gaussian of every (tile, depth) list entry, the tile of every list, and the lists' starts and lengths."""
    a, b, c = var
    alpha, u, v = rec[:, 5], rec[:, 0], rec[:, 1]
    mid = 0.5 * (a + c)
    radius = 3.0 * torch.sqrt(mid + torch.sqrt((mid * mid - (a * c - b * b)).clamp(min=0.0)))
    L2 = 2.0 * torch.log(255.0 * alpha.clamp(min=1e-30)).clamp(min=0.0)
    ex = torch.minimum(radius, torch.sqrt(L2 * a) * 1.0001 + 0.01)
    ey = torch.minimum(radius, torch.sqrt(L2 * c) * 1.0001 + 0.01)
    tx, ty = (cam.width + tw - 1) // tw, (cam.height + th - 1) // th
    x0, x1 = ((u - ex) / tw).floor().clamp(0, tx), (((u + ex) / tw).floor() + 1).clamp(0, tx)
    y0, y1 = ((v - ey) / th).floor().clamp(0, ty), (((v + ey) / th).floor() + 1).clamp(0, ty)
    ok = (alpha >= 1.0 / 255.0) & (z > float(torch.tensor(cam.znear, dtype=torch.float32))) & (x0 < x1) & (y0 < y1)
    vis = ok.nonzero()[:, 0]
    vis = vis[torch.argsort(z[vis], stable=True)]
    w, h = (x1 - x0)[vis].long(), (y1 - y0)[vis].long()
    g = torch.repeat_interleave(vis, w * h)
    first = torch.repeat_interleave(torch.cumsum(w * h, 0) - w * h, w * h)
    local = torch.arange(g.numel(), device=g.device) - first
    ww = torch.repeat_interleave(w, w * h)
    tile = (y0[g].long() + local // ww) * tx + x0[g].long() + local % ww
    order = torch.argsort(tile, stable=True)
    tiles, counts = torch.unique_consecutive(tile[order], return_counts=True)
    return g[order], tiles, torch.cumsum(counts, 0) - counts, counts


def _blend(rec, z, var, cam, tw, th, grad):
    """The image of one view (3, H, W) and, with grad(image) = dL/dC, the gradient of its records."""
    dev, H, W = rec.device, cam.height, cam.width
    tx, ty = (W + tw - 1) // tw, (H + th - 1) // th
    image = torch.tensor(BG, dtype=torch.float64, device=dev)[:, None, None].expand(3, ty * th, tx * tw).clone()
    view = image.view(3, ty, th, tx, tw)
    ids, tiles, start, count = _tile_lists(rec.detach(), z.detach(), var, cam, tw, th)
    px = torch.arange(tw * th, device=dev)
    by = torch.argsort(count, descending=True)
    leaf = rec.detach()
    drec = torch.zeros_like(leaf)
    sizes = count[by].tolist()

    def chunks():
        i = 0
        while i < len(sizes):
            m = max(1, (3 << 24) // (sizes[i] * tw * th))
            yield by[i:i + m], sizes[i]
            i += m

    def composite(t, longest, table):
        at = start[t][:, None] + torch.arange(longest, device=dev)
        live = torch.arange(longest, device=dev) < count[t][:, None]
        e = ids[at.clamp(max=ids.numel() - 1)]
        r = table[e]
        X = ((tiles[t] % tx) * tw)[:, None] + px % tw + 0.5
        Y = ((tiles[t] // tx) * th)[:, None] + px // tw + 0.5
        dx, dy = r[..., 0, None] - X[:, None], r[..., 1, None] - Y[:, None]
        power = -0.5 * (r[..., 2, None] * dx * dx + r[..., 4, None] * dy * dy) - r[..., 3, None] * dx * dy
        al = (r[..., 5, None] * torch.exp(power))
        keep = (al >= 1.0 / 255.0) & live[..., None]
        al = torch.where(keep, al.clamp(max=0.99), torch.zeros_like(al))
        after = torch.cumprod(1.0 - al.detach(), 1)
        al = torch.where(after < 1e-4, torch.zeros_like(al), al)
        # T before each entry, as the exponential of a running sum of logarithms (its reverse is cheap and exact enough)
        run = torch.cumsum(torch.log1p(-al), 1)
        before = torch.exp(run - torch.log1p(-al))
        C = torch.einsum("tlp,tlc->tcp", al * before, r[..., 6:9])
        bg = torch.tensor(BG, dtype=torch.float64, device=dev)
        return C + bg[None, :, None] * torch.exp(run[:, -1])[:, None], e, live

    for t, longest in chunks():
        with torch.no_grad():
            C = composite(t, longest, leaf)[0]
        view[:, tiles[t] // tx, :, tiles[t] % tx] = C.view(-1, 3, th, tw)
    image = image[:, :H, :W].contiguous()
    if grad is None:
        return image, None
    dC = torch.zeros(3, ty * th, tx * tw, dtype=torch.float64, device=dev)
    dC[:, :H, :W] = grad(image)
    dview = dC.view(3, ty, th, tx, tw)
    for t, longest in chunks():
        table = leaf.clone().requires_grad_()
        C, _, _ = composite(t, longest, table)
        want = dview[:, tiles[t] // tx, :, tiles[t] % tx].reshape(-1, 3, th * tw)
        drec += torch.autograd.grad(C, table, want)[0]
    return image, drec


def exact(case, seed):
    p = {k: v.double() for k, v in _scene(case, seed).items()}
    if case["kind"] == "cache":
        A, Sdi, Sc = _slice_state(p)
        iu = torch.triu_indices(3, 3)
        return torch.cat([A.reshape(-1, 9).T, Sdi[:, iu[0], iu[1]].T, Sc.reshape(-1, 9).T,
                          torch.sigmoid(p["opacity_logit"])[None]])
    if case["kind"] == "axes":
        # an axis has no sign of its own, so the rotation has no one value
        scale = torch.linalg.eigvalsh(_slice_state(p)[2].cpu()).clamp(min=0.0).sqrt().flip(1).T.contiguous()
        return {"rotation": None, "scale": scale}
    train, infer = case["kind"] == "train", case["kind"] == "infer"
    cams = _cameras(case)
    total = 3 * sum(c.width * c.height for c in cams)
    given = None if infer else _images(case, seed, train).double()
    images, loss, at = [], torch.zeros(1, dtype=torch.float64, device="cuda"), 0
    sums = {k: torch.zeros_like(v) for k, v in p.items()}
    for cam in cams:
        m = 3 * cam.width * cam.height
        mine = None if infer else given[at:at + m].view(3, cam.height, cam.width)
        at += m
        leaves = {k: v.clone().requires_grad_(not infer) for k, v in p.items()}
        rec, z, var = _records(leaves, _slice_state(leaves), cam, case["degree"])
        grad = None if infer else (lambda im, mine=mine: torch.sign(im - mine) / total) if train else (lambda im, mine=mine: mine)
        image, drec = _blend(rec, z, var, cam, 16, case["tile_h"], grad)
        images.append(image.reshape(-1))
        if train:
            loss += (image - mine).abs().sum() / total
        if drec is not None:
            seen = (drec != 0).any(1)               # a Gaussian behind the camera has no finite record
            g = torch.autograd.grad(rec[seen], list(leaves.values()), drec[seen])
            for k, v in zip(leaves, g):
                sums[k] += torch.nan_to_num(v)
    images = torch.cat(images)
    if infer:
        return images
    out = {"images": images, "grads": sums}
    return dict(out, loss=loss) if train else out
