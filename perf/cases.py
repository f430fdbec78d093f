"""Performance cases of the splatting library: what a mapping or tracking program
asks of it, from a 2,000-Gaussian render to a 4M-Gaussian mapping step.

Kinds of case (the framework's public entry points in each):

* ``autograd``  ``rasterize`` and its backward inside a user's own loss: the
  differentiable render of one or a few small keyframes, all gradients and the
  pose twist.
* ``render``    ``Rasterizer.forward``: a novel view, no gradients.
* ``tracking``  ``TrackingStep.run``: one pose-only iteration against a sensor
  frame with its keypoints.
* ``mapping``   ``MappingStep.run``: one joint iteration over a window of
  keyframes with Adam on every Gaussian.
* ``loss``      ``gs_loss_l1`` + ``gs_loss_ssim`` on images the caller rendered.
* ``upkeep``    the calls made when a keyframe enters the map: densification,
  pruning, compaction of parameters and optimiser state, spatial order.
* ``decode``    ``gs_decode_keyframes``: sensor frames to loss targets.

Scenes are indoor rooms with boxes (Gaussians on the surfaces, in the Morton
order a maintained map is stored in); sensor images are ray-cast from the same
rooms, so the maps are near their targets as in a running session.  Learning
rates are those of a late iteration (a hundredth of the defaults): a step moves
its own state, and the work must stay what it was over many steps.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2405_19614_gb300 as gs
from paper_2405_19614_gb300.pipeline import DEFAULT_LR, PARAM_ORDER, MappingStep, TrackingStep

DEV = "cuda"
DEPTH_UNIT = 1.0 / 5000.0  # metres per unit of a 16-bit sensor depth
NEAR, BLUR = 0.2, 0.3
TAU = 0.005  # pruning threshold
UNEVEN = "640x480*4,960x540*4,1200x680*4,1280x720*4"


def _case(name, kind, n, sizes, **more):
    c = dict(name=name, kind=kind, n=n, sizes=sizes, degree=3, scene="room6x5", focal=0.0, tile_w=16, tile_h=16,
             zeta=0.0, keypoints=0, w_c=1.0, w_d=0.5, gate=False)
    c.update(more)
    return c


def listed():
    return [
        # the smallest differentiable render: a toy scene, where launches and latency are everything
        _case("autograd-2k-64x48", "autograd", 2000, "64x48", degree=0, scene="cube", focal=60.0),
        # a user's own loss over three cropped frames of odd sizes, a submap of moderate size
        _case("autograd-20k-3odd", "autograd", 20011, "321x243,283x197,401x301", degree=2, scene="room4x4"),
        # a novel view for display
        _case("render-300k-1200x680", "render", 300_000, "1200x680", focal=600.0),
        # pose refinement of a VGA sensor frame, the inner loop of tracking (about 100 of these a frame)
        _case("tracking-100k-640x480", "tracking", 100_000, "640x480", scene="room4x4", focal=525.0, keypoints=1000,
              w_c=0.5, w_d=1.0, gate=True),
        # mapping with one keyframe, L1 losses only
        _case("mapping-300k-1200x680", "mapping", 300_000, "1200x680", focal=600.0, w_d=0.1),
        # the window of eight keyframes with the whole mapping loss (tile shape as the autotuner picks it)
        _case("mapping-1M-8x1200x680", "mapping", 1_000_000, "1200x680*8", focal=600.0, zeta=0.3, keypoints=1000,
              tile_w=32, tile_h=16),
        # a long session: a whole floor, sixteen keyframes of four cameras
        _case("mapping-4M-16-uneven", "mapping", 4_000_000, UNEVEN, scene="floor30x20", zeta=0.3, keypoints=1000),
        # the mapping loss on a caller's own renders, odd image sizes
        _case("loss-4x641x479", "loss", 0, "641x479*4", scene="room4x4", focal=525.0, zeta=0.3),
        # a keyframe enters a map of a million Gaussians
        _case("upkeep-1M-640x480", "upkeep", 1_000_000, "640x480", focal=525.0),
        # the keyframes of a mapping window arrive from the sensor
        _case("decode-8x1200x680", "decode", 0, "1200x680*8"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["autograd", "render", "tracking", "mapping", "mapping", "loss", "upkeep", "decode"])
    if kind == "decode":
        w = _log_int(rng, 64, 1280)
        return _drawn(_case("", kind, 0, f"{w}x{_log_int(rng, 48, 720)}*{rng.randint(1, 8)}"))
    w = _log_int(rng, 64, 1280)
    h = max(33, int(w * rng.uniform(0.5, 0.8)))
    views = 1 if kind in ("render", "tracking", "upkeep") else rng.randint(1, 8 if kind == "mapping" else 4)
    sizes = f"{w}x{h}*{views}"
    if views > 1 and rng.random() < 0.4:  # cameras of different sizes
        sizes = ",".join(f"{max(33, w - rng.randint(0, w // 3))}x{max(33, h - rng.randint(0, h // 3))}"
                         for _ in range(views))
    focal = w * rng.uniform(0.5, 0.9)
    n = {"autograd": (2000, 300_000), "render": (2000, 1_000_000), "tracking": (10_000, 300_000),
         "mapping": (5000, 1_500_000), "loss": (1, 1), "upkeep": (20_000, 2_000_000)}[kind]
    more = dict(scene=rng.choice(["room4x4", "room6x5", "floor30x20"]), focal=focal)
    if kind in ("autograd", "render"):
        more["degree"] = rng.randint(0, 3)
    if kind == "tracking":
        more.update(scene="room4x4", keypoints=rng.randint(200, 2000), w_c=0.5, w_d=1.0, gate=True)
    if kind == "mapping":
        tw, th = rng.choice([(16, 16), (16, 16), (32, 16), (32, 32), (8, 8), (64, 32)])
        more.update(zeta=rng.choice([0.0, 0.3]), keypoints=rng.choice([0, 1000]), tile_w=tw, tile_h=th)
    if kind == "loss":
        more.update(zeta=0.3, gate=rng.random() < 0.3)
    return _drawn(_case("", kind, 0 if kind == "loss" else _log_int(rng, *n), sizes, **more))


def _drawn(c):
    c.pop("name")
    return c


def _sizes(case):
    out = []
    for part in case["sizes"].split(","):
        wh, _, k = part.partition("*")
        w, h = wh.split("x")
        out += [(int(w), int(h))] * int(k or 1)
    return out


def _intr(case):
    return [[float(np.float32(case["focal"] or w / 2.0))] * 2 + [w / 2.0, h / 2.0] for w, h in _sizes(case)]


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

ROOMS = {"room4x4": ((4.0, 4.0, 3.0), 12), "room6x5": ((6.0, 5.0, 3.0), 20), "floor30x20": ((30.0, 20.0, 3.0), 60)}


def _boxes(case, seed):
    """The room as (lo, hi) boxes: the first seen from inside, the others (furniture, partition walls) from outside."""
    (X, Y, Z), count = ROOMS.get(case["scene"], ROOMS["room4x4"])
    r = random.Random(seed)
    boxes = [((-X / 2, -Y / 2, 0.0), (X / 2, Y / 2, Z))]
    for _ in range(count):
        sx, sy, sz = r.uniform(0.2, 1.0), r.uniform(0.2, 1.0), r.uniform(0.2, 1.1)
        cx = r.uniform(-X / 2 + 0.3 + sx / 2, X / 2 - 0.3 - sx / 2)
        cy = r.uniform(-Y / 2 + 0.3 + sy / 2, Y / 2 - 0.3 - sy / 2)
        boxes.append(((cx - sx / 2, cy - sy / 2, 0.0), (cx + sx / 2, cy + sy / 2, sz)))
    if X > 20:  # 3 x 2 rooms with door gaps
        for x in (-X / 6, X / 6):
            for y0 in (-Y / 2, 0.0):
                boxes.append(((x - 0.1, y0, 0.0), (x + 0.1, y0 + Y / 4 - 0.6, Z)))
                boxes.append(((x - 0.1, y0 + Y / 4 + 0.6, 0.0), (x + 0.1, y0 + Y / 2, Z)))
        for x0 in (-X / 2, -X / 6, X / 6):
            boxes.append(((x0, -0.1, 0.0), (x0 + X / 6 - 0.6, 0.1, Z)))
            boxes.append(((x0 + X / 6 + 0.6, -0.1, 0.0), (x0 + X / 3, 0.1, Z)))
    return boxes


def _paint(p):
    """Surface colour in [0, 1] at world points p [., 3]."""
    x, y, z = p.unbind(-1)
    return torch.stack([0.5 + 0.25 * torch.sin(2.1 * x + 1.3 * z) + 0.1 * torch.sin(9.0 * y + 4.0 * z),
                        0.5 + 0.25 * torch.sin(1.7 * y - 1.1 * z + 1.0) + 0.1 * torch.sin(8.0 * x + 5.0 * z),
                        0.5 + 0.25 * torch.sin(1.3 * x + 1.9 * y + 2.0) + 0.1 * torch.sin(7.0 * z + 6.0 * x)], -1)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _morton(m):
    lo, hi = m.min(0).values, m.max(0).values
    q = ((m - lo) / (hi - lo).clamp_min(1e-9) * 1023.0).long()
    code = torch.zeros(len(m), dtype=torch.int64, device=m.device)
    for b in range(10):
        for a in range(3):
            code |= ((q[:, a] >> b) & 1) << (3 * b + a)
    return torch.argsort(code, stable=True)


def _gaussians(case, seed):
    """The map: Gaussian parameters as device tensors."""
    n, K, g = case["n"], (case["degree"] + 1) ** 2, _gen(seed)
    rand = lambda *s: torch.rand(*s, generator=g, device=DEV)  # noqa: E731
    randn = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    C0 = 0.5 / math.sqrt(math.pi)
    if case["scene"] == "cube":
        means = rand(n, 3) * 2.0 + torch.tensor([-1.0, -1.0, 2.0], device=DEV)
        ls = -3.5 + 0.5 * randn(n, 3)
        logit, colour = randn(n), rand(n, 3)
    else:
        faces, areas = [], []
        for k, (lo, hi) in enumerate(_boxes(case, seed)):
            d = [hi[a] - lo[a] for a in range(3)]
            for ax in range(3):
                for at in (lo[ax], hi[ax]):
                    if k and ax == 2 and at == 0.0:
                        continue  # the face on the floor
                    faces.append((ax, at, lo, d))
                    areas.append(d[0] * d[1] * d[2] / d[ax])
        fid = torch.searchsorted(torch.cumsum(torch.tensor(areas, device=DEV), 0),
                                 rand(n) * sum(areas)).clamp_max(len(faces) - 1)
        lo = torch.tensor([f[2] for f in faces], device=DEV)[fid]
        d = torch.tensor([f[3] for f in faces], device=DEV)[fid]
        means = lo + rand(n, 3) * d
        ax = torch.tensor([f[0] for f in faces], device=DEV)[fid]
        means.scatter_(1, ax[:, None], (torch.tensor([f[1] for f in faces], device=DEV)[fid] + 0.01 * randn(n))[:, None])
        means = means[_morton(means)]
        ls = math.log(min(0.06, max(0.015, 0.64 * math.sqrt(sum(areas) / n)))) + 0.3 * randn(n, 3)
        logit, colour = 1.0 + randn(n), _paint(means)
    sh = 0.1 * randn(n, K, 3)
    sh[:, 0] = (colour - 0.5) / C0 + (0.02 * randn(n, 3) if K > 1 else 0.0)
    q = randn(n, 4)
    q /= q.norm(dim=1, keepdim=True)
    return dict(means=means.contiguous(), log_scales=ls, quats=q, opacity_logit=logit, sh=sh, sh_degree=case["degree"])


def _poses(case, seed):
    """World-to-camera [V, 12]: an arc through the room at eye height (a cube is seen from the origin)."""
    V = len(_sizes(case))
    if case["scene"] == "cube":
        return torch.eye(4, device=DEV)[:3].reshape(1, 12).repeat(V, 1).contiguous()
    (X, Y, _), _ = ROOMS[case["scene"]]
    r = random.Random(seed + 1)
    centre, rad = ((X / 3, Y / 4), 2.5) if X > 20 else ((r.uniform(-0.3, 0.3), r.uniform(-0.3, 0.3)), 0.25 * min(X, Y))
    a0, out = r.uniform(0, 2 * math.pi), []
    for k in range(V):
        a = a0 + 0.35 * k
        eye = np.array([centre[0] + rad * math.cos(a), centre[1] + rad * math.sin(a), 1.5 + 0.1 * math.sin(a)])
        yaw, pitch = a + math.pi / 2 + 0.3 * math.sin(0.7 * k), -0.1 + 0.05 * math.cos(k)
        f = np.array([math.cos(yaw) * math.cos(pitch), math.sin(yaw) * math.cos(pitch), math.sin(pitch)])
        right = np.cross(f, [0.0, 0.0, 1.0])
        right /= np.linalg.norm(right)
        R = np.stack([right, np.cross(f, right), f])
        out.append(np.concatenate([R, (-R @ eye)[:, None]], 1).reshape(12))
    return torch.from_numpy(np.stack(out).astype(np.float32)).to(DEV)


def _sensor(case, seed, viewmats, holes=0.0, noise=1.0):
    """Ray-cast colour [P, 3] and depth [P] of the room with sensor noise; holes: share of pixels without depth."""
    boxes, rgbs, depths = _boxes(case, seed), [], []
    for (w, h), (fx, fy, cx, cy), E in zip(_sizes(case), _intr(case), viewmats.cpu().double().reshape(-1, 3, 4)):
        R, t = E[:, :3], E[:, 3]
        o = (-R.T @ t).tolist()
        y, x = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")
        c = torch.stack([(x + 0.5 - cx) / fx, (y + 0.5 - cy) / fy, torch.ones_like(x, dtype=torch.float32)], -1)
        d = (c.reshape(-1, 1, 3) * R.T.float().to(DEV)).sum(-1)
        d = torch.where(d.abs() < 1e-7, torch.full_like(d, 1e-7), d)
        inv = 1.0 / d
        z = None
        for k, (lo, hi) in enumerate(boxes):
            t1 = torch.stack([(lo[a] - o[a]) * inv[:, a] for a in range(3)], -1)
            t2 = torch.stack([(hi[a] - o[a]) * inv[:, a] for a in range(3)], -1)
            near, far = torch.minimum(t1, t2).amax(-1), torch.maximum(t1, t2).amin(-1)
            z = far if k == 0 else torch.where((near < far) & (near > 0.05) & (near < z), near, z)
        rgbs.append(_paint(torch.tensor(o, device=DEV, dtype=torch.float32) + d * z[:, None]))
        depths.append(z)
    g = _gen(seed + 7)
    rgb, z = torch.cat(rgbs), torch.cat(depths)
    rgb = (rgb + 0.02 * noise * torch.randn(rgb.shape, generator=g, device=DEV)).clamp(0, 1)
    z = z + 0.005 * noise * torch.randn(z.shape, generator=g, device=DEV)
    if holes:
        z = torch.where(torch.rand(z.shape, generator=g, device=DEV) < holes, torch.zeros_like(z), z)
    return rgb.contiguous(), z.contiguous()


def _keypoints(case, seed, viewmats, depth):
    """Map points back-projected from the sensor depth, observed with one pixel of noise."""
    if not case["keypoints"]:
        return None
    g, pts, obs, ids, base = _gen(seed + 9), [], [], [], 0
    for v, ((w, h), (fx, fy, cx, cy)) in enumerate(zip(_sizes(case), _intr(case))):
        m = case["keypoints"]
        px = torch.randint(8, w - 8, (m,), generator=g, device=DEV)
        py = torch.randint(8, h - 8, (m,), generator=g, device=DEV)
        z = depth[base + py * w + px].double().clamp_min(0.5)
        E = viewmats[v].double().reshape(3, 4)
        pc = torch.stack([(px + 0.5 - cx) / fx * z, (py + 0.5 - cy) / fy * z, z], -1) - E[:, 3]
        pts.append((pc[:, :, None] * E[:, :3]).sum(1).float())  # R^T (p - t)
        obs.append(torch.stack([px + 0.5, py + 0.5], -1).float() + torch.randn(m, 2, generator=g, device=DEV))
        ids.append(torch.full((m,), v, dtype=torch.int32, device=DEV))
        base += w * h
    return dict(points=torch.cat(pts).contiguous(), obs=torch.cat(obs).contiguous(), view_ids=torch.cat(ids))


def _moved(viewmats, seed, trans=0.01, rot=math.radians(0.5)):
    """Poses off by a centimetre and half a degree: where tracking starts."""
    r = np.random.RandomState(seed)
    out = []
    for E in viewmats.cpu().double().numpy().reshape(-1, 3, 4):
        a, b = r.standard_normal(3), r.standard_normal(3)
        a, b = a / np.linalg.norm(a) * trans, b / np.linalg.norm(b)
        Kx = np.array([[0, -b[2], b[1]], [b[2], 0, -b[0]], [-b[1], b[0], 0]])
        R = np.eye(3) + math.sin(rot) * Kx + (1 - math.cos(rot)) * Kx @ Kx
        out.append(np.concatenate([R @ E[:, :3], (R @ E[:, 3] + a)[:, None]], 1).reshape(12))
    return torch.from_numpy(np.stack(out).astype(np.float32)).to(DEV)


def _upstream(case, seed):
    """Image gradients of a mean L1 loss over colour, depth and border mask."""
    P, g = sum(w * h for w, h in _sizes(case)), _gen(seed + 3)
    s = lambda *k: torch.randint(0, 2, k, generator=g, device=DEV).float() * 2 - 1  # noqa: E731
    return s(P, 3) / (3 * P), 0.5 * s(P) / P, 0.1 * s(P) / P


def _renders(case, seed):
    """A caller's renders of the sensor frames: the frames without their noise, with the errors of an unfinished map."""
    vm = _poses(case, seed)
    t_rgb, t_z = _sensor(case, seed, vm, holes=0.03 if case["gate"] else 0.0)
    g = _gen(seed + 5)
    rgb, z = _sensor(case, seed, vm, noise=0.0)
    rgb = (0.97 * rgb + 0.01 + 0.01 * torch.randn(rgb.shape, generator=g, device=DEV)).clamp(0, 1)
    z = z + 0.02 * torch.randn(z.shape, generator=g, device=DEV)
    alpha = 0.97 + 0.03 * torch.rand(z.shape, generator=g, device=DEV)
    return rgb.contiguous(), z.contiguous(), alpha, t_rgb, t_z


def _upkeep_inputs(case, seed):
    p, vm = _gaussians(case, seed), _poses(case, seed)
    p["opacity_logit"] = p["opacity_logit"] - 2.5  # a share of the map has faded below the threshold
    rgb, z = _sensor(case, seed, vm, holes=0.05)
    x = torch.arange(len(z), device=DEV)
    # the part of the frame the map does not cover yet: a broad border and scattered gaps
    alpha = 0.5 + 0.4 * torch.sin(x * 0.011 + seed) + 0.25 * torch.rand(len(z), generator=_gen(seed + 2), device=DEV)
    return p, vm, rgb, z, alpha.clamp(0, 1)


def _frames(case, seed):
    P, g = sum(w * h for w, h in _sizes(case)), _gen(seed)
    rgb8 = torch.randint(0, 256, (P, 3), generator=g, device=DEV, dtype=torch.uint8)
    d16 = torch.randint(0, 30000, (P,), generator=g, device=DEV, dtype=torch.int16)
    return rgb8, torch.where(d16 < 1500, torch.zeros_like(d16), d16)


# --------------------------------------------------------------------------
# prepare, run
# --------------------------------------------------------------------------

def prepare(case, seed):
    kind, tile = case["kind"], (case["tile_w"], case["tile_h"])
    s = dict(kind=kind)
    if kind == "decode":
        s["rgb8"], s["d16"] = _frames(case, seed)
        P = s["d16"].numel()
        s["rgb"], s["depth"] = torch.empty(P, 3, device=DEV), torch.empty(P, device=DEV)
        return s
    if kind == "loss":
        s["rgb"], s["depth"], s["alpha"], s["t_rgb"], s["t_z"] = _renders(case, seed)
        P = s["depth"].numel()
        s["views"] = gs.make_views(_intr(case), _sizes(case))
        s["case"] = case
        s["loss"], s["d_rgb"], s["d_z"] = torch.zeros(1, device=DEV), torch.empty(P, 3, device=DEV), torch.empty(P, device=DEV)
        s["ws"] = torch.empty(gs.gs_ssim_workspace_size(P), dtype=torch.uint8, device=DEV)
        return s
    if kind == "upkeep":
        p, vm, rgb, z, alpha = _upkeep_inputs(case, seed)
        n, P, K = case["n"], z.numel(), (case["degree"] + 1) ** 2
        grown = {k: torch.zeros(n + P, *p[k].shape[1:], device=DEV) for k in PARAM_ORDER}
        for k in PARAM_ORDER:
            grown[k][:n] = p[k]
        s.update(n=n, views=gs.make_views(_intr(case), _sizes(case)), vm=vm, rgb=rgb, z=z, alpha=alpha,
                 grown=dict(grown, sh_degree=case["degree"]), state={k: p[k].reshape(n, -1) for k in PARAM_ORDER})
        g = _gen(seed + 4)
        for name in ("m", "v"):  # optimiser state
            for k in PARAM_ORDER:
                s["state"][f"{name}.{k}"] = torch.randn(s["state"][k].shape, generator=g, device=DEV)
        s["kept"] = {k: torch.zeros_like(x) for k, x in s["state"].items()}
        i32 = lambda m: torch.zeros(m, dtype=torch.int32, device=DEV)  # noqa: E731
        s.update(index=i32(n), order=i32(n), n_kept=i32(1), n_added=i32(1), status=i32(1),
                 ws=torch.empty(gs.gs_select_workspace_size(max(n, P)), dtype=torch.uint8, device=DEV),
                 ows=torch.empty(gs.gs_spatial_order_workspace_size(n), dtype=torch.uint8, device=DEV))
        return s
    vm = _poses(case, seed)
    intr, sizes = _intr(case), _sizes(case)
    # room for the pairs: small maps have large splats
    pairs = 8 * case["n"] * len(sizes) + 64 * min(case["n"], 100_000) * len(sizes) + (1 << 20)
    if kind == "mapping":
        n, K = case["n"], (case["degree"] + 1) ** 2
        t_rgb, t_z = _sensor(case, seed, vm)
        shapes = dict(means=(n, 3), log_scales=(n, 3), quats=(n, 4), opacity_logit=(n,), sh=(n, K, 3))
        step = MappingStep(dict({k: np.zeros(x, np.float32) for k, x in shapes.items()}, sh_degree=case["degree"]),
                           intr, sizes, vm.cpu().numpy(), t_rgb, t_z, w_c=case["w_c"], w_d=case["w_d"],
                           keypoints=_keypoints(case, seed, vm, t_z), zeta=case["zeta"], tile=tile,
                           pair_capacity=pairs, lrs={k: 0.01 * x for k, x in DEFAULT_LR.items()})
        p = _gaussians(case, seed)
        for k in PARAM_ORDER:
            step.params[k].copy_(p[k])
        s["step"] = step
        s["m"], s["v"] = step.flat.views(step.m), step.flat.views(step.v)
        return s
    p = _gaussians(case, seed)
    if kind == "tracking":
        t_rgb, t_z = _sensor(case, seed, vm, holes=0.05)
        s["step"] = TrackingStep(p, intr, sizes, _moved(vm, seed).cpu().numpy(), t_rgb, t_z,
                                 keypoints=_keypoints(case, seed, vm, t_z), w_c=case["w_c"], w_d=case["w_d"],
                                 pair_capacity=pairs, tile=tile)
        return s
    s.update(params=p, vm=vm, rast=gs.Rasterizer(case["n"], case["degree"], intr, sizes, pairs, tile=tile))
    if kind == "autograd":
        for k in PARAM_ORDER:
            p[k].requires_grad_(True)
        s["twist"] = torch.zeros(len(sizes), 6, device=DEV, requires_grad=True)
        s["up"] = _upstream(case, seed)
    return s


def run(s):
    kind = s["kind"]
    if kind == "render":
        img = s["rast"].forward(s["params"], s["vm"])
        return {k: img[k] for k in ("rgb", "depth", "alpha")}
    if kind == "autograd":
        p = s["params"]
        rgb, depth, alpha = gs.rasterize(s["rast"], p, s["vm"], s["twist"])
        inputs = [p[k] for k in PARAM_ORDER] + [s["twist"]]
        grads = torch.autograd.grad([rgb, depth, alpha], inputs, list(s["up"]))
        return dict(rgb=rgb, depth=depth, alpha=alpha, grads=dict(zip(PARAM_ORDER + ("twist",), grads)))
    if kind == "mapping":
        st = s["step"]
        st.run()
        img = st.rast.img
        tensors = lambda d: {k: d[k] for k in PARAM_ORDER}  # noqa: E731
        return dict(loss=st.loss, rgb=img["rgb"], depth=img["depth"], alpha=img["alpha"], twist=st.d_twist,
                    grads=tensors(st.grads), params=tensors(st.params), m=tensors(s["m"]), v=tensors(s["v"]))
    if kind == "tracking":
        st = s["step"]
        st.run()
        img = st.rast.img
        return dict(loss=st.loss, rgb=img["rgb"], depth=img["depth"], alpha=img["alpha"], d_twist=st.d_twist,
                    poses=st.viewmats)
    if kind == "loss":
        c = s["case"]
        k1 = 1.0 - c["zeta"]
        s["loss"].zero_()
        gs.gs_loss_l1(s["rgb"], s["depth"], s["alpha"], s["t_rgb"], s["t_z"], k1 * c["w_c"], k1 * c["w_d"], c["gate"],
                      0.99, s["loss"], s["d_rgb"], s["d_z"])
        gs.gs_loss_ssim(s["rgb"], s["t_rgb"], s["views"], c["zeta"], s["loss"], s["d_rgb"], s["ws"])
        return dict(loss=s["loss"], d_rgb=s["d_rgb"], d_depth=s["d_z"])
    if kind == "upkeep":
        gs.gs_densify(s["alpha"], s["rgb"], s["z"], s["views"], s["vm"], 0.5, 0.0, s["grown"], s["n"],
                      s["n"] + s["z"].numel(), s["n_added"], s["ws"], s["status"])
        gs.gs_prune_select(s["state"]["opacity_logit"], TAU, s["index"], s["n_kept"], s["ws"])
        gs.gs_compact_rows(s["index"], [(s["state"][k], s["kept"][k]) for k in s["state"]])
        gs.gs_spatial_order(s["state"]["means"], s["order"], s["ows"], s["status"])
        return dict(n_added=s["n_added"], n_kept=s["n_kept"], index=s["index"], order=s["order"],
                    grown={k: s["grown"][k] for k in PARAM_ORDER}, kept=s["kept"])
    gs.gs_decode_keyframes(s["rgb8"], s["d16"], DEPTH_UNIT, s["rgb"], s["depth"])
    return dict(rgb=s["rgb"], depth=s["depth"])


def work(case):
    """Bytes: inputs once, outputs once.  Flops: the compositing's evaluations and
    blends (about 3600 a pixel forward and 5100 backward on covered indoor
    views), the SSIM windows (about 700 a pixel)."""
    kind, n, K, V = case["kind"], case["n"], (case["degree"] + 1) ** 2, len(_sizes(case))
    P, per = sum(w * h for w, h in _sizes(case)), 4 * (11 + 3 * K)
    if kind == "decode":
        return dict(bytes=21 * P, flops=4 * P)
    if kind == "loss":
        return dict(bytes=(36 + 16) * P, flops=720 * P)
    if kind == "upkeep":
        return dict(bytes=n * (4 + 3 * per + 0.55 * 3 * per + 12 + 8) + P * (20 + 0.45 * per), flops=n + P)
    if kind == "render":
        return dict(bytes=n * per + 20 * P, flops=3600 * P)
    if kind == "tracking":
        return dict(bytes=n * per + 36 * P + 20 * case["keypoints"], flops=8700 * P)
    if kind == "autograd":
        return dict(bytes=2 * n * per + 40 * P, flops=8700 * P)
    return dict(bytes=n * 7 * per + 36 * P + 20 * V * case["keypoints"], flops=(8700 + (700 if case["zeta"] else 0)) * P)


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------

def _sh_basis(d, degree):
    x, y, z = d.unbind(-1)
    pi = math.pi
    c1 = math.sqrt(3 / (4 * pi))
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if degree > 0:
        Y += [c1 * y, c1 * z, c1 * x]
    if degree > 1:
        a, b, c = math.sqrt(15 / pi) / 2, math.sqrt(5 / pi) / 4, math.sqrt(15 / pi) / 4
        Y += [a * x * y, a * y * z, b * (3 * z * z - 1), a * x * z, c * (x * x - y * y)]
    if degree > 2:
        a, b = math.sqrt(35 / (2 * pi)) / 4, math.sqrt(105 / pi) / 2
        c, d_, e = math.sqrt(21 / (2 * pi)) / 4, math.sqrt(7 / pi) / 4, math.sqrt(105 / pi) / 4
        Y += [a * y * (3 * x * x - y * y), b * x * y * z, c * y * (5 * z * z - 1), d_ * z * (5 * z * z - 3),
              c * x * (5 * z * z - 1), e * z * (x * x - y * y), a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _project64(p, E, xi, intr, size, degree):
    """Splats of one view: (u, v, z, conic, log opacity, colour), radius; differentiable in p and the twist xi."""
    fx, fy, cx, cy = intr
    w, h = size
    rho, phi = xi[:3], xi[3:]
    zero = torch.zeros((), dtype=torch.float64, device=DEV)
    X = torch.stack([torch.stack([zero, -phi[2], phi[1]]), torch.stack([phi[2], zero, -phi[0]]),
                     torch.stack([-phi[1], phi[0], zero])])
    R, t = E[:, :3], E[:, 3]
    R, t = R + X @ R, t + rho + X @ t  # first order in the twist, which is zero
    pc = p["means"] @ R.T + t
    x, y, z = pc.unbind(-1)
    zs = torch.where(z > NEAR, z, torch.ones_like(z))
    lx, ly = 1.3 * 0.5 * w / fx, 1.3 * 0.5 * h / fy
    tx, ty = (x / zs).clamp(-lx, lx), (y / zs).clamp(-ly, ly)
    q = p["quats"] / p["quats"].norm(dim=1, keepdim=True)
    qw, a, b, c = q.unbind(-1)
    rot = torch.stack([1 - 2 * (b * b + c * c), 2 * (a * b - qw * c), 2 * (a * c + qw * b),
                       2 * (a * b + qw * c), 1 - 2 * (a * a + c * c), 2 * (b * c - qw * a),
                       2 * (a * c - qw * b), 2 * (b * c + qw * a), 1 - 2 * (a * a + b * b)], -1).reshape(-1, 3, 3)
    M = rot * torch.exp(p["log_scales"])[:, None, :]
    zero_ = torch.zeros_like(zs)
    J = torch.stack([fx / zs, zero_, -fx * tx / zs, zero_, fy / zs, -fy * ty / zs], -1).reshape(-1, 2, 3)
    T = (J @ R) @ M
    S = T @ T.transpose(1, 2)
    ca, cb, cc = S[:, 0, 0] + BLUR, S[:, 0, 1], S[:, 1, 1] + BLUR
    det = ca * cc - cb * cb
    mid = 0.5 * (ca + cc)
    radius = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp_min(0)))).detach()
    radius = torch.where((z > NEAR) & (det > 0), radius, torch.zeros_like(radius))
    d = p["means"] + R.T @ t  # minus the camera centre
    Y = _sh_basis(d / d.norm(dim=1, keepdim=True), degree)
    colour = ((Y[:, :, None] * p["sh"]).sum(1) + 0.5).clamp_min(0)
    logo = torch.nn.functional.logsigmoid(p["opacity_logit"])
    return [fx * x / zs + cx, fy * y / zs + cy, z, cc / det, -cb / det, ca / det, logo] + list(colour.unbind(-1)), radius


def _composite64(rec, px, py):
    """rec [10][T, L, 1] front to back, pixels [T, 1, A]: colour, depth and border mask [T, A, .]."""
    u, v, z, A, B, C, lo = rec[:7]
    dx, dy = px - u, py - v
    l = lo - 0.5 * (A * dx * dx + C * dy * dy) - B * dx * dy
    alpha = torch.exp(l).clamp_max(0.99)
    alpha = torch.where(alpha.detach() >= 1.0 / 255.0, alpha, torch.zeros_like(alpha))
    logT = torch.cumsum(torch.log1p(-alpha), 1)
    T = torch.exp(logT)
    before = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
    wgt = torch.where(T.detach() >= 1e-4, alpha * before, torch.zeros_like(T))
    return [(wgt * c).sum(1) for c in rec[7:10]] + [(wgt * z).sum(1), wgt.sum(1)]


def _render64(case, p, E, grad_of=None):
    """Images of all views and, with grad_of(images) -> image gradients, the
    gradients with respect to the parameters and the twists."""
    tw, th = case["tile_w"], case["tile_h"]
    leaves = {k: p[k].detach().double().requires_grad_(grad_of is not None) for k in PARAM_ORDER}
    xi = torch.zeros(len(E), 6, dtype=torch.float64, device=DEV, requires_grad=grad_of is not None)
    chunks, images = [], []
    with torch.set_grad_enabled(grad_of is not None):
        splats = [_project64(leaves, E[v].double().reshape(3, 4), xi[v], k, s, case["degree"])
                  for v, (k, s) in enumerate(zip(_intr(case), _sizes(case)))]
    recs = []
    for v, ((w, h), (sp, radius)) in enumerate(zip(_sizes(case), splats)):
        u, vv, z = (x.detach() for x in sp[:3])
        nx, ny = -(-w // tw), -(-h // th)
        x0, x1 = ((torch.floor((u + sgn * radius) / tw)).clamp(-1, nx) for sgn in (-1, 1))
        y0, y1 = ((torch.floor((vv + sgn * radius) / th)).clamp(-1, ny) for sgn in (-1, 1))
        ok = (radius > 0) & (x1 >= 0) & (y1 >= 0) & (x0 < nx) & (y0 < ny)
        x0, y0, x1, y1 = x0.clamp_min(0).long(), y0.clamp_min(0).long(), x1.clamp_max(nx - 1).long(), y1.clamp_max(ny - 1).long()
        ids = torch.nonzero(ok).flatten()
        ids = ids[torch.argsort(z[ids], stable=True)]
        nw, nh = (x1 - x0 + 1)[ids], (y1 - y0 + 1)[ids]
        rep = torch.repeat_interleave(torch.arange(len(ids), device=DEV), nw * nh)
        k = torch.arange(len(rep), device=DEV) - (torch.cumsum(nw * nh, 0) - nw * nh)[rep]
        tile = (y0[ids][rep] + k // nw[rep]) * nx + x0[ids][rep] + k % nw[rep]
        order = torch.argsort(tile, stable=True)
        entry = ids[rep[order]]
        count = torch.bincount(tile, minlength=nx * ny)
        start = torch.cumsum(count, 0) - count
        rec = torch.stack([x.detach() for x in sp])
        recs.append(rec.requires_grad_(grad_of is not None))
        by_len = torch.argsort(count, descending=True).tolist()
        counts, at = count.tolist(), 0
        while at < len(by_len):
            L = max(1, counts[by_len[at]])
            m = max(1, min(len(by_len) - at, 24_000_000 // (L * tw * th)))
            tl = torch.tensor(by_len[at:at + m], device=DEV)
            at += m
            j = torch.arange(L, device=DEV)
            valid = j[None] < count[tl][:, None]
            e = torch.where(valid, entry[(start[tl][:, None] + j[None]).clamp_max(max(0, len(entry) - 1))] if len(entry)
                            else torch.zeros_like(valid, dtype=torch.int64), 0)
            a = torch.arange(tw * th, device=DEV)
            px, py = (tl % nx)[:, None] * tw + (a % tw)[None], (tl // nx)[:, None] * th + (a // tw)[None]
            chunks.append((v, e, valid, px, py, (px < w) & (py < h)))
        images.append(torch.zeros(w * h, 5, dtype=torch.float64, device=DEV))

    def composite(c):
        v, e, valid, px, py, inside = c
        r = recs[v][:, e][..., None]
        parts = [x for x in r]
        parts[6] = torch.where(valid[..., None], parts[6], torch.full_like(parts[6], -1e3))
        out = _composite64(parts, (px + 0.5).double()[:, None], (py + 0.5).double()[:, None])
        at = (py * _sizes(case)[v][0] + px)[inside]
        return torch.stack([o[inside] for o in out], -1), at

    with torch.no_grad():
        for c in chunks:
            out, at = composite(c)
            images[c[0]][at] = out
    img = torch.cat(images)
    img = dict(rgb=img[:, :3], depth=img[:, 3], alpha=img[:, 4])
    if grad_of is None:
        return img
    up = grad_of(img)
    up = torch.cat([up[0].double(), up[1].double()[:, None], (torch.zeros_like(img["alpha"]) if up[2] is None else up[2].double())[:, None]], 1)
    base = np.concatenate([[0], np.cumsum([w * h for w, h in _sizes(case)])])
    acc = [torch.zeros_like(r) for r in recs]
    for c in chunks:
        with torch.enable_grad():
            out, at = composite(c)
            acc[c[0]] += torch.autograd.grad(out, recs[c[0]], up[int(base[c[0]]) + at])[0]
    outs, ups = [], []
    for (sp, _), a in zip(splats, acc):
        outs += sp
        ups += list(a)
    g = torch.autograd.grad(outs, [leaves[k] for k in PARAM_ORDER] + [xi], ups)
    return img, dict(zip(PARAM_ORDER, g[:5])), g[5]


def _l1_64(case, img, t_rgb, t_z, w_c, w_d, gate):
    """The L1 losses and their image gradients."""
    P = len(t_z)
    rc, rz = img["rgb"] - t_rgb.double(), img["depth"] - t_z.double()
    G = ((t_z > 0) & (img["depth"] > 0) & (img["alpha"] > 0.99)).double() if gate else torch.ones(P, dtype=torch.float64, device=DEV)
    loss = w_c / (3 * P) * (G[:, None] * rc.abs()).sum() + w_d / P * (G * rz.abs()).sum()
    return loss, w_c / (3 * P) * G[:, None] * torch.sign(rc), w_d / P * G * torch.sign(rz)


def _ssim_64(case, rgb, t_rgb, weight):
    """weight (1 - mean SSIM) over all views and its gradient (11 x 11 Gaussian window, sigma 1.5, zero padding)."""
    i = torch.arange(11, dtype=torch.float64, device=DEV) - 5
    g = torch.exp(-i * i / 4.5)
    g = (g / g.sum()).tolist()

    def window(m):
        for dim in (0, 1):
            n = m.shape[dim]
            pad = torch.nn.functional.pad(m, (0, 0, 0, 0, 5, 5) if dim == 0 else (0, 0, 5, 5))
            m = sum(g[k] * pad.narrow(dim, k, n) for k in range(11))
        return m

    x = rgb.detach().double().requires_grad_(True)
    total, base = 0.0, 0
    with torch.enable_grad():
        for w, h in _sizes(case):
            X, Y = x[base:base + w * h].view(h, w, 3), t_rgb[base:base + w * h].double().view(h, w, 3)
            mx, my = window(X), window(Y)
            vx, vy, vxy = window(X * X) - mx * mx, window(Y * Y) - my * my, window(X * Y) - mx * my
            total = total + ((2 * mx * my + 1e-4) * (2 * vxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (vx + vy + 9e-4))).sum()
            base += w * h
        loss = weight * (1 - total / x.numel())
    return loss.detach(), torch.autograd.grad(loss, x)[0]


def _reproj_64(case, kp, E, weight):
    """The keypoint re-projection loss and its twist gradient."""
    xi = torch.zeros(len(E), 6, dtype=torch.float64, device=DEV, requires_grad=True)
    if kp is None:
        return 0.0, torch.zeros_like(xi)
    v = kp["view_ids"].long()
    k = torch.tensor(_intr(case), dtype=torch.float64, device=DEV)[v]
    M = E.double().reshape(-1, 3, 4)[v]
    with torch.enable_grad():
        p = (M[:, :, :3] * kp["points"].double()[:, None, :]).sum(-1) + M[:, :, 3]
        p = p + xi[v, :3] + torch.linalg.cross(xi[v, 3:], p)
        ok = p[:, 2].detach() > NEAR
        z = torch.where(ok, p[:, 2], torch.ones_like(p[:, 2]))
        r = kp["obs"].double() - torch.stack([k[:, 0] * p[:, 0] / z + k[:, 2], k[:, 1] * p[:, 1] / z + k[:, 3]], -1)
        loss = weight / len(v) * (r.norm(dim=1) * ok).sum()
    return loss.detach(), torch.autograd.grad(loss, xi)[0]


def _pose_step_64(E, g, lr=(5e-4, 3e-4)):
    """The first Adam step on each twist, folded into the pose: Exp(xi) E."""
    xi = -torch.tensor([lr[0]] * 3 + [lr[1]] * 3, dtype=torch.float64, device=DEV) * g / (g.abs() + 1e-15)
    out = []
    for M, x in zip(E.double().reshape(-1, 3, 4), xi):
        A = torch.zeros(4, 4, dtype=torch.float64, device=DEV)
        A[0, 1], A[0, 2], A[1, 0], A[1, 2], A[2, 0], A[2, 1] = -x[5], x[4], x[5], -x[3], -x[4], x[3]
        A[:3, 3] = x[:3]
        X = torch.linalg.matrix_exp(A)
        out.append(torch.cat([X[:3, :3] @ M[:, :3], (X[:3, :3] @ M[:, 3] + X[:3, 3])[:, None]], 1).reshape(12))
    return torch.stack(out)


def exact(case, seed):
    kind = case["kind"]
    P = sum(w * h for w, h in _sizes(case))
    if kind == "decode":
        rgb8, d16 = _frames(case, seed)
        return dict(rgb=rgb8.double() / 255.0, depth=d16.double() * float(np.float32(DEPTH_UNIT)))
    if kind == "loss":
        rgb, z, alpha, t_rgb, t_z = _renders(case, seed)
        k1 = 1.0 - case["zeta"]
        loss, d_rgb, d_z = _l1_64(case, dict(rgb=rgb.double(), depth=z.double(), alpha=alpha), t_rgb, t_z,
                                  k1 * case["w_c"], k1 * case["w_d"], case["gate"])
        more, d_more = _ssim_64(case, rgb, t_rgb, case["zeta"])
        return dict(loss=(loss + more).reshape(1), d_rgb=d_rgb + d_more, d_depth=d_z)
    if kind == "upkeep":
        return _exact_upkeep(case, seed)
    if P > 2_500_000 or case["n"] > 400_000:
        return None  # the large windows take over 20 seconds in 64 bits
    p, vm = _gaussians(case, seed), _poses(case, seed)
    if kind == "render":
        return _render64(case, p, vm)
    if kind == "autograd":
        img, g, xi = _render64(case, p, vm, lambda _: _upstream(case, seed))
        return dict(img, grads=dict(g, twist=xi))
    out = {}
    t_rgb, t_z = _sensor(case, seed, vm, holes=0.05 if kind == "tracking" else 0.0)
    kp = _keypoints(case, seed, vm, t_z)
    if kind == "tracking":
        vm = _moved(vm, seed)

    def losses(img):
        k1 = 1.0 - case["zeta"]
        out["loss"], d_rgb, d_z = _l1_64(case, img, t_rgb, t_z, k1 * case["w_c"], k1 * case["w_d"], case["gate"])
        if case["zeta"]:
            more, d_more = _ssim_64(case, img["rgb"], t_rgb, case["zeta"])
            out["loss"], d_rgb = out["loss"] + more, d_rgb + d_more
        return d_rgb, d_z, None

    img, g, xi = _render64(case, p, vm, losses)
    more, d_xi = _reproj_64(case, kp, vm, 1.5)
    loss, xi = (out["loss"] + more).reshape(1), xi + d_xi
    if kind == "tracking":
        return dict(img, loss=loss, d_twist=xi.reshape(-1), poses=_pose_step_64(vm, xi))
    lr = {k: 0.01 * DEFAULT_LR[k] for k in PARAM_ORDER}
    new = {k: p[k].double() - lr[k] * g[k] / (g[k].abs() + 1e-15) for k in PARAM_ORDER}
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    return dict(img, loss=loss, twist=xi, grads=g, params=new, m={k: (1 - b1) * g[k] for k in PARAM_ORDER},
                v={k: (1 - b2) * g[k] ** 2 for k in PARAM_ORDER})


def _exact_upkeep(case, seed):
    p, vm, rgb, z, alpha = _upkeep_inputs(case, seed)
    n, (w, h), (fx, fy, cx, cy) = case["n"], _sizes(case)[0], _intr(case)[0]
    at = torch.nonzero((alpha < 0.5) & (z > 0)).flatten()
    E, d = vm[0].double().reshape(3, 4), z[at].double()
    pc = torch.stack([((at % w) + 0.5 - cx) / fx * d, ((at // w) + 0.5 - cy) / fy * d, d], -1) - E[:, 3]
    grown, m = {}, len(at)
    for k in PARAM_ORDER:
        grown[k] = torch.zeros(n + len(z), *p[k].shape[1:], dtype=torch.float64, device=DEV)
        grown[k][:n] = p[k].double()
    grown["means"][n:n + m] = (pc[:, :, None] * E[:, :3]).sum(1)
    grown["log_scales"][n:n + m] = torch.log(d / fx)[:, None]
    grown["quats"][n:n + m, 0] = 1.0
    grown["sh"][n:n + m, 0] = (rgb[at].double() - 0.5) * (2.0 * math.sqrt(math.pi))
    keep = p["opacity_logit"] >= float(np.float32(math.log(TAU / (1.0 - TAU))))
    state, g = {k: p[k].reshape(n, -1) for k in PARAM_ORDER}, _gen(seed + 4)
    for name in ("m", "v"):
        for k in PARAM_ORDER:
            state[f"{name}.{k}"] = torch.randn(state[k].shape, generator=g, device=DEV)
    kept = {}
    for k, x in state.items():
        kept[k] = torch.zeros(x.shape, dtype=torch.float64, device=DEV)
        kept[k][:int(keep.sum())] = x[keep].double()
    return dict(n_added=None, n_kept=None, index=None, order=None, grown=grown, kept=kept)
