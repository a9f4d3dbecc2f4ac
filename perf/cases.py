"""Performance cases of the rasterizer: the calls a user of this package makes, over the range of maps and
image sizes they are made on.

A case is a dict of plain values: ``op`` names the call, the other entries its sizes and types. Scenes are
drawn on the GPU from a seed with the distributions of the repository's own workloads: free Gaussians in a
box, Gaussians on planes crossing the frustum, a room, an aerial site (ground, boxes and large translucent
splats), cameras walking through them. Key-frames are smooth images with sensor noise.

``exact`` computes what ``run`` returns in 64 bits with plain torch, from the definitions: EWA projection
with a 0.3 px^2 dilation, 16 x 16 tiles inside the 3-sigma rectangle, front-to-back compositing in depth
order, the L1 loss, and reverse mode through all of it.
"""
import math

import torch

from paper_2509_06433_gb300 import api, autograd, autotune
from paper_2509_06433_gb300.tracking import MappingStep, Tracker

DEV = "cuda"
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
NEAR, LAMBDA = 0.2, 0.1
PARAMS = ("means", "log_scales", "quats", "opacity_logits", "rgb")


def listed():
    return [
        # the smallest render: a preview of a young map (all Gaussians in front of the camera)
        {"name": "render_small", "op": "render", "scene": "free", "N": 10_000, "K": 1, "W": 320, "H": 240, "f": 300.0,
         "dtype": "f32"},
        # a headset frame of the interactive viewer: a stereo pair at the camera's 672 x 376
        {"name": "render_stereo", "op": "render", "scene": "planes", "N": 100_000, "K": 2, "W": 672, "H": 376,
         "f": 336.0, "dtype": "f32"},
        # one viewpoint of a large reduced-storage site map
        {"name": "render_aerial", "op": "render", "scene": "aerial", "N": 2_000_000, "K": 1, "W": 1280, "H": 720,
         "f": 900.0, "dtype": "f16"},
        # a single-view mapping iteration, replayed as a graph, kernel variants tuned as the benchmark does
        {"name": "map_single", "op": "map", "scene": "planes", "N": 100_000, "K": 1, "W": 640, "H": 480, "f": 525.0,
         "dtype": "f32", "tune": True},
        # the online mapper's iteration over its window of 4 key-frames, library-chosen variants (the
        # online mapper does not tune)
        {"name": "map_online", "op": "map", "scene": "room", "N": 40_000, "K": 4, "W": 672, "H": 376, "f": 260.0,
         "dtype": "f32", "tune": False},
        # a mapping window of 8 key-frames over a BF16 room
        {"name": "map_window", "op": "map", "scene": "room", "N": 500_000, "K": 8, "W": 640, "H": 480, "f": 525.0,
         "dtype": "bf16", "tune": True},
        # the largest: 16 key-frames over a 2M-Gaussian FP16 site
        {"name": "map_aerial", "op": "map", "scene": "aerial", "N": 2_000_000, "K": 16, "W": 1280, "H": 720,
         "f": 900.0, "dtype": "f16", "tune": True},
        # one pose-tracking iteration (pose-only backward and the on-device pose step), as a graph
        {"name": "track", "op": "track", "scene": "planes", "N": 300_000, "K": 1, "W": 640, "H": 480, "f": 525.0,
         "dtype": "f32"},
        # a differentiable render with view-dependent colour inside a torch training loop, called eagerly,
        # on an image that fills no whole number of tiles
        {"name": "autograd_sh3", "op": "autograd", "scene": "planes", "N": 60_000, "K": 1, "W": 501, "H": 333,
         "f": 420.0, "dtype": "f32", "sh": 3},
        # the optimiser step of a large map: FP32 masters and moments, FP16 storage refreshed
        {"name": "adam", "op": "adam", "N": 2_000_000, "dtype": "f16", "sh": -1},
        # map accuracy of a window's four key-frames: PSNR and SSIM with its map
        {"name": "metrics", "op": "metrics", "B": 4, "W": 672, "H": 376},
        # the sort primitive on (tile, depth) keys of a 640 x 480 view
        {"name": "sort_pairs", "op": "sort", "n": 850_000, "bits": 43},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["render", "render", "map", "map", "map", "track", "autograd", "adam", "metrics", "sort"])
    if op == "adam":
        return {"op": op, "N": _log(rng, 20_000, 2_000_000), "dtype": rng.choice(["f32", "bf16", "f16"]),
                "sh": rng.choice([-1, -1, 1])}
    if op == "metrics":
        return {"op": op, "B": rng.randint(1, 8), "W": rng.randint(160, 1280), "H": rng.randint(120, 720)}
    if op == "sort":
        return {"op": op, "n": _log(rng, 5_000, 4_000_000), "bits": rng.randint(33, 56)}
    W, H = rng.randint(160, 1280), rng.randint(120, 720)
    c = {"op": op, "scene": rng.choice(["free", "planes", "room", "aerial"]), "N": _log(rng, 10_000, 2_000_000), "K": 1,
         "W": W, "H": H, "f": round(W * rng.uniform(0.5, 0.95), 1), "dtype": "f32"}
    if op == "render":
        c["K"] = rng.randint(1, 4)
        c["dtype"] = rng.choice(["f32", "bf16", "f16"])
    elif op == "map":
        c["K"] = rng.randint(1, 16)
        most = 32_000_000 if c["scene"] == "aerial" else 4_000_000  # elsewhere most of the map is in every view
        c["N"] = min(c["N"], most // c["K"])
        c["dtype"] = rng.choice(["f32", "bf16", "f16"])
        c["tune"] = rng.random() < 0.5
    elif op == "autograd":
        c["sh"] = rng.choice([-1, 1, 2, 3])
        c["N"] = min(c["N"], 300_000)
    return c


# ------------------------------------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 13)


def _uni(gen, n, lo, hi):
    lo, hi = torch.tensor(lo, device=DEV), torch.tensor(hi, device=DEV)
    return lo + (hi - lo) * torch.rand((n, 3), generator=gen, device=DEV)


def _quat_mul(a, b):
    aw, ax, ay, az = a.unbind(-1)
    bw, bx, by, bz = b.unbind(-1)
    return torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                        aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], -1)


def _rotation(q):
    """Rotation matrices of unit quaternions (w, x, y, z)."""
    w, x, y, z = q.unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).unflatten(-1, (3, 3))


def _free(gen, n, lo, hi, ls=(-3.0, 0.5), logit=(0.0, 1.0)):
    r = lambda *s: torch.randn(s, generator=gen, device=DEV)  # noqa: E731
    return [_uni(gen, n, lo, hi), ls[0] + ls[1] * r(n, 3), torch.nn.functional.normalize(r(n, 4), dim=1),
            logit[0] + logit[1] * r(n)]


def _plane(gen, n, center, frame, half, inplane=(-3.0, 0.5)):
    """n flat Gaussians on planes: centres [n, 3], frame quaternions [n, 4] (third axis = the normal), half
    extents [n, 2] in the plane."""
    r = lambda *s: torch.randn(s, generator=gen, device=DEV)  # noqa: E731
    ab = (2 * torch.rand((n, 2), generator=gen, device=DEV) - 1) * half
    R = _rotation(frame)
    means = center + ab[:, :1] * R[:, :, 0] + ab[:, 1:] * R[:, :, 1]
    th = math.pi * torch.rand(n, generator=gen, device=DEV)
    spin = torch.stack([torch.cos(th), torch.zeros_like(th), torch.zeros_like(th), torch.sin(th)], -1)
    ls = torch.cat([inplane[0] + inplane[1] * r(n, 2), -6.0 + 0.3 * r(n, 1)], 1)
    return [means, ls, _quat_mul(frame, spin), r(n)]


def _axis_quat(axis, deg):
    h = math.radians(deg) / 2
    v = {"x": (1, 0, 0), "y": (0, 1, 0), "z": (0, 0, 1)}[axis]
    return torch.tensor([math.cos(h)] + [math.sin(h) * a for a in v], device=DEV)


def _scene(kind, n, seed):
    """means, log-scales, quaternions, opacity logits, colours, drawn on the GPU."""
    gen = _gen(seed)
    if kind == "free":
        parts = [_free(gen, n, (-2.0, -2.0, 2.0), (2.0, 2.0, 8.0))]
    elif kind == "planes":  # half free, half on three planes crossing the frustum
        m = n - n // 2
        which = torch.arange(m, device=DEV) % 3
        centers = _uni(gen, 3, (-1.0, -1.0, 3.5), (1.0, 1.0, 6.5))
        frames = torch.nn.functional.normalize(torch.randn((3, 4), generator=gen, device=DEV), dim=1)
        parts = [_free(gen, n // 2, (-2.0, -2.0, 2.0), (2.0, 2.0, 8.0)),
                 _plane(gen, m, centers[which], frames[which], torch.full((m, 2), 2.5, device=DEV))]
    elif kind == "room":  # the six walls of an 8 x 6 x 3 m room and 10% free
        X, Y, Z = 8.0, 6.0, 3.0
        walls = [((X / 2, Y / 2, 0), _axis_quat("x", 0), (X / 2, Y / 2)), ((X / 2, Y / 2, Z), _axis_quat("x", 180), (X / 2, Y / 2)),
                 ((X / 2, 0, Z / 2), _axis_quat("x", -90), (X / 2, Z / 2)), ((X / 2, Y, Z / 2), _axis_quat("x", 90), (X / 2, Z / 2)),
                 ((0, Y / 2, Z / 2), _axis_quat("y", 90), (Z / 2, Y / 2)), ((X, Y / 2, Z / 2), _axis_quat("y", -90), (Z / 2, Y / 2))]
        area = torch.tensor([a * b for _, _, (a, b) in walls], device=DEV)
        m = n - n // 10
        which = torch.multinomial(area, m, replacement=True, generator=gen)
        parts = [_free(gen, n // 10, (0.3, 0.3, 0.3), (X - 0.3, Y - 0.3, Z - 0.3)),
                 _plane(gen, m, torch.tensor([w[0] for w in walls], device=DEV)[which], torch.stack([w[1] for w in walls])[which],
                        torch.tensor([w[2] for w in walls], device=DEV)[which])]
    else:  # aerial: ground, the tops and sides of 40 boxes, 20% large translucent
        large, half = n // 5, 40.0
        ground = (n - large) // 2
        m = n - large - ground
        one = torch.ones(40, device=DEV)
        rnd = lambda lo, hi: lo + (hi - lo) * torch.rand(40, generator=gen, device=DEV)  # noqa: E731
        cx, cy, sx, sy, h, yaw = rnd(-35, 35), rnd(-35, 35), rnd(2, 8), rnd(2, 8), rnd(2, 10), rnd(0, 2 * math.pi)
        q = torch.stack([torch.cos(yaw / 2), 0 * one, 0 * one, torch.sin(yaw / 2)], -1)
        z = 0 * one
        faces = [((z, z, h), ("x", 0), (sx / 2, sy / 2)), ((sx / 2, z, h / 2), ("y", 90), (h / 2, sy / 2)),
                 ((-sx / 2, z, h / 2), ("y", -90), (h / 2, sy / 2)), ((z, sy / 2, h / 2), ("x", -90), (sx / 2, h / 2)),
                 ((z, -sy / 2, h / 2), ("x", 90), (sx / 2, h / 2))]
        center = torch.stack([(_rotation(q) @ torch.stack(c, -1)[:, :, None])[:, :, 0] for c, _, _ in faces], 1)
        center = center + torch.stack([cx, cy, z], -1)[:, None]
        frame = torch.stack([_quat_mul(q, _axis_quat(*a).expand(40, 4)) for _, a, _ in faces], 1)
        size = torch.stack([torch.stack(s, -1) for _, _, s in faces], 1)
        which = torch.arange(m, device=DEV) % 200
        up = torch.tensor([1.0, 0, 0, 0], device=DEV).expand(ground, 4)
        parts = [_plane(gen, ground, torch.zeros((ground, 3), device=DEV), up, torch.full((ground, 2), half, device=DEV),
                        (-4.0, 0.7)),
                 _plane(gen, m, center.reshape(-1, 3)[which], frame.reshape(-1, 4)[which], size.reshape(-1, 2)[which],
                        (-4.0, 0.7)),
                 _free(gen, large, (-half, -half, 0.0), (half, half, 8.0), (-2.0, 0.5), (-1.0, 1.0))]
    out = [torch.cat([p[i] for p in parts]).contiguous() for i in range(4)]
    return out + [torch.rand((n, 3), generator=gen, device=DEV)]


def _cameras(c, seed):
    """[K, 16] cameras: at the origin along z (a few centimetres apart) for the box scenes, a walk inside the
    room, a flight over the site with a 20 degree down-tilt."""
    rnd = torch.Generator().manual_seed(int(seed) * 31 + 7)
    u = lambda lo, hi: lo + (hi - lo) * torch.rand((), generator=rnd, dtype=torch.float64).item()  # noqa: E731
    rows = []
    kind, W, H, f = c["scene"], c["W"], c["H"], c["f"]
    pos = [4.0, 3.0, 1.5] if kind == "room" else [u(-20, 20), u(-20, 20), u(3, 10)]
    yaw, tilt = u(0, 2 * math.pi), math.radians(20.0) if kind == "aerial" else 0.0
    for k in range(c["K"]):
        if kind in ("free", "planes"):
            R, t = torch.eye(3, dtype=torch.float64), torch.tensor([-0.064 * k, 0.0, 0.0], dtype=torch.float64)
        else:
            d = torch.tensor([math.cos(yaw) * math.cos(tilt), math.sin(yaw) * math.cos(tilt), -math.sin(tilt)],
                             dtype=torch.float64)
            r = torch.linalg.cross(torch.tensor([0, 0, -1.0], dtype=torch.float64), d)
            r = r / r.norm()
            R = torch.stack([r, torch.linalg.cross(d, r), d])
            t = -R @ torch.tensor(pos, dtype=torch.float64)
            yaw += math.radians(u(-10, 10))
            step = 0.3 if kind == "room" else 0.5
            nxt = [pos[0] + step * math.cos(yaw), pos[1] + step * math.sin(yaw), pos[2]]
            if kind == "aerial":
                nxt[2] = min(10.0, max(3.0, nxt[2] + u(-0.3, 0.3)))
            elif not (0.8 < nxt[0] < 7.2 and 0.8 < nxt[1] < 5.2):
                yaw, nxt = yaw + math.pi, [2 * pos[0] - nxt[0], 2 * pos[1] - nxt[1], pos[2]]
            pos = nxt
        rows.append(torch.cat([torch.tensor([f, f, W / 2, H / 2], dtype=torch.float64), R.reshape(9), t]))
    return torch.stack(rows).float().to(DEV).contiguous()


def _frames(c, seed):
    """Key-frames [K,3,H,W] and depths [K,H,W]: smooth fields plus sensor noise."""
    gen = _gen(seed + 101)
    K, H, W = c["K"], c["H"], c["W"]
    low = torch.rand((K, 4, H // 32 + 2, W // 32 + 2), generator=gen, device=DEV)
    img = torch.nn.functional.interpolate(low, size=(H, W), mode="bilinear", align_corners=False)
    img = img + 0.02 * torch.randn(img.shape, generator=gen, device=DEV)
    return img[:, :3].clamp(0, 1).contiguous(), (1.0 + 8.0 * img[:, 3].clamp(0, 1)).contiguous()


def _sensor_noise(c, seed):
    gen = _gen(seed + 303)
    K, H, W = c["K"], c["H"], c["W"]
    return [0.01 * torch.randn(s, generator=gen, device=DEV) for s in ((K, 3, H, W), (K, H, W))]


def _off_pose(cams, seed):
    """The poses turned by 2 degrees and moved by 5 cm, in random directions."""
    rnd = torch.Generator().manual_seed(int(seed) * 17 + 3)
    out = cams.double().cpu()
    for cam in out:
        a, d = (torch.nn.functional.normalize(torch.randn(3, generator=rnd, dtype=torch.float64), dim=0) for _ in range(2))
        S = torch.tensor([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]], dtype=torch.float64)
        th = math.radians(2.0)
        dR = torch.eye(3, dtype=torch.float64) + math.sin(th) * S + (1 - math.cos(th)) * S @ S
        cam[4:13] = (dR @ cam[4:13].view(3, 3)).reshape(9)
        cam[13:16] = dR @ cam[13:16] + 0.05 * d
    return out.float().to(DEV).contiguous()


def _sh(n, degree, seed):
    gen = _gen(seed + 55)
    f = 0.15 * torch.randn((n, (degree + 1) ** 2, 3), generator=gen, device=DEV)
    f[:, 0] = 2 * torch.rand((n, 3), generator=gen, device=DEV) - 1
    return f


def _map_arrays(c, seed):
    """The Gaussians in their storage types (means stay FP32)."""
    p = _scene(c["scene"], c["N"], seed)
    if c.get("sh", -1) >= 0:
        p[4] = _sh(c["N"], c["sh"], seed)
    dt = DTYPES[c["dtype"]]
    return [p[0]] + [t.to(dt) for t in p[1:]]


def _upstream(c, seed):
    gen = _gen(seed + 77)
    K, H, W = c["K"], c["H"], c["W"]
    return [(torch.rand(s, generator=gen, device=DEV) - 0.5) / (H * W) for s in ((K, 3, H, W), (K, H, W), (K, H, W))]


def _adam_inputs(c, seed):
    """A map's masters, gradients and mid-run moments (the 200th step)."""
    gen = _gen(seed)
    width = 3 * max(1, (c["sh"] + 1) ** 2)
    n = c["N"]
    shapes = {"means": (n, 3), "log_scales": (n, 3), "quats": (n, 4), "opacity_logits": (n,),
              "rgb": (n, 3) if c["sh"] < 0 else (n, width // 3, 3)}
    rnd = lambda s: torch.randn(s, generator=gen, device=DEV)  # noqa: E731
    masters = {k: rnd(s) for k, s in shapes.items()}
    grads = {k: 1e-6 * rnd(s) for k, s in shapes.items()}
    seen = torch.rand(n, generator=gen, device=DEV) < 0.6  # Gaussians outside every view have zero gradients
    for k, g in grads.items():
        g *= seen.view(-1, *([1] * (g.dim() - 1)))
    total = n * (11 + width)
    m = 3e-7 * torch.randn(total, generator=gen, device=DEV)
    v = 1e-12 * (0.05 + torch.rand(total, generator=gen, device=DEV))
    return masters, grads, torch.cat([m, v, torch.tensor([200.0], device=DEV)])


def _images(c, seed):
    gen = _gen(seed)
    low = torch.rand((c["B"], 3, c["H"] // 16 + 2, c["W"] // 16 + 2), generator=gen, device=DEV)
    x = torch.nn.functional.interpolate(low, size=(c["H"], c["W"]), mode="bilinear", align_corners=False)
    y = (x + 0.05 * torch.randn(x.shape, generator=gen, device=DEV)).clamp(0, 1)
    return x.contiguous(), y.contiguous()


def _sort_inputs(c, seed):
    gen = _gen(seed)
    n, bits = c["n"], c["bits"]
    hi = torch.randint(0, 1 << (bits - 32), (n,), generator=gen, device=DEV)
    depth = (0.2 + 8.0 * torch.rand(n, generator=gen, device=DEV)).view(torch.int32).long()
    return (hi << 32) | depth, torch.arange(n, dtype=torch.int32, device=DEV)


# ------------------------------------------------------------------------------------------------ the calls

def prepare(case, seed):
    c, op = case, case["op"]
    if op == "adam":
        masters, grads, state = _adam_inputs(c, seed)
        dt = DTYPES[c["dtype"]]
        g = api.Gaussians(masters["means"], *(masters[k].to(dt) for k in PARAMS[1:]))
        opt = api.MapOptimizer(g)
        for k in PARAMS:  # the masters of a map in training hold more than its storage does
            getattr(opt.masters, k).copy_(masters[k])
        opt.state.copy_(state)
        return {"case": c, "opt": opt, "grads": grads, "g": g, "n": state.numel() // 2}
    if op == "metrics":
        x, y = _images(c, seed)
        return {"case": c, "x": x, "y": y, "map": torch.empty_like(x)}
    if op == "sort":
        keys, vals = _sort_inputs(c, seed)
        tmp = torch.empty(max(256, api.gs_sort_pairs_tmp_size(c["n"])), dtype=torch.uint8, device=DEV)
        return {"case": c, "k0": keys, "v0": vals, "keys": keys.clone(), "vals": vals.clone(), "tmp": tmp}
    g = api.Gaussians(*_map_arrays(c, seed))
    cams = _cameras(c, seed)
    if op == "track":  # the observed frame: the map from the true pose; tracking starts 2 degrees and 5 cm off
        r = api.Rasterizer(c["W"], c["H"], c["K"], c["N"])
        r.plan(g, cams)
        seen = r.render(g, cams)
        n_rgb, n_depth = _sensor_noise(c, seed)
        start = _off_pose(cams, seed)
        return {"case": c, "tracker": Tracker(g, start, c["W"], c["H"], seen["rgb"] + n_rgb, seen["depth"] + n_depth)}
    sh = c.get("sh", -1)
    r = api.Rasterizer(c["W"], c["H"], c["K"], c["N"], pair_capacity=max(1 << 16, c["N"] * c["K"]),
                       sh_degree=sh if sh >= 0 else None)
    r.plan(g, cams)
    s = {"case": c, "r": r, "g": g, "cams": cams}
    if op == "render":
        s["out"] = r.new_outputs()
    elif op == "map":
        if c["tune"]:
            autotune.tune(r, g, cams, reps=3)
        s["step"] = MappingStep(r, g, cams, *_frames(c, seed))
    else:
        s["leaves"] = [getattr(g, k).requires_grad_() for k in PARAMS]
        s["xi"] = torch.zeros((c["K"], 6), device=DEV, requires_grad=True)
        s["up"] = _upstream(c, seed)
    return s


def run(state):
    s, op = state, state["case"]["op"]
    if op == "render":
        return s["r"].render(s["g"], s["cams"], s["out"])
    if op == "map":
        m = s["step"]
        m.replay()
        return {"grads": m.grads, "loss": m.loss, **m.out}
    if op == "track":
        t = s["tracker"]
        return {"cams": t.run(1), "pose_grad": t.pose_grad, "loss": t.loss}
    if op == "autograd":
        out = autograd.render(s["r"], *s["leaves"], s["cams"], s["xi"])
        grads = torch.autograd.grad(out, [*s["leaves"], s["xi"]], s["up"])
        return {"out": list(out), "grads": list(grads)}
    if op == "adam":
        o = s["opt"]
        o.step(s["grads"])
        return {"masters": [getattr(o.masters, k) for k in PARAMS], "storage": [getattr(s["g"], k) for k in PARAMS],
                "m": o.state[:s["n"]], "v": o.state[s["n"]:-1], "steps": o.state[-1:]}
    if op == "metrics":
        return {"psnr": api.gs_psnr(s["x"], s["y"]), "ssim": api.gs_ssim(s["x"], s["y"], ssim_map=s["map"]),
                "map": s["map"]}
    # the sort is in place: a frame's keys are written by the copies, then sorted
    s["keys"].copy_(s["k0"])
    s["vals"].copy_(s["v0"])
    api.gs_sort_pairs(s["keys"], s["vals"], s["case"]["bits"], s["tmp"])
    return {"keys": s["keys"], "vals": s["vals"]}


def work(case):
    """Bytes: inputs and outputs once. Operations: about 80 splats blended per covered pixel, 11 operations
    each forwards and 44 backwards, and about 600 per (view, Gaussian) in the projection and its backward."""
    c, op = case, case["op"]
    if op == "sort":
        return {"bytes": 2 * 12 * c["n"], "flops": 0}
    if op == "metrics":
        px = c["B"] * 3 * c["H"] * c["W"]
        return {"bytes": 12 * px, "flops": px * (5 * 11 * 2 * 2 + 25)}
    w = 3 * max(1, (c.get("sh", -1) + 1) ** 2)
    store = torch.empty((), dtype=DTYPES[c["dtype"]]).element_size()
    n = c["N"]
    if op == "adam":
        return {"bytes": n * (11 + w) * (4 * 7) + (n * (8 + w) * store if store < 4 else 0), "flops": n * (11 + w) * 12}
    px = c["K"] * c["H"] * c["W"]
    read = n * (12 + (8 + w) * store)
    if op == "render":
        return {"bytes": read + 24 * px, "flops": px * 80 * 11 + 300 * n * c["K"]}
    if op == "track":
        return {"bytes": read + (16 + 24) * px, "flops": px * 80 * 55 + 600 * n * c["K"]}
    return {"bytes": read + n * (11 + w) * 4 + (16 + 24) * px, "flops": px * 80 * 55 + 600 * n * c["K"]}


# ------------------------------------------------------------------------------------------- in 64 bits

def _sh_colour(f, d):
    """max(sum_i Y_i(d) f_i + 1/2, 0), real harmonics with the Condon-Shortley phase, bands 0 to 3."""
    x, y, z = d.unbind(-1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if f.shape[1] > 1:
        a = math.sqrt(3 / (4 * pi))
        Y += [-a * y, a * z, -a * x]
    if f.shape[1] > 4:
        a, b, e = math.sqrt(15 / (4 * pi)), math.sqrt(5 / (16 * pi)), math.sqrt(15 / (16 * pi))
        Y += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z, e * (x * x - y * y)]
    if f.shape[1] > 9:
        a, b, e = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi)), math.sqrt(21 / (32 * pi))
        h, k = math.sqrt(7 / (16 * pi)), math.sqrt(105 / (16 * pi))
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -e * y * (4 * z * z - x * x - y * y),
              h * z * (2 * z * z - 3 * x * x - 3 * y * y), -e * x * (4 * z * z - x * x - y * y), k * z * (x * x - y * y),
              -a * x * (x * x - 3 * y * y)]
    return (torch.einsum("ni,nic->nc", torch.stack(Y, -1), f) + 0.5).clamp_min(0)


def _project(P, cam, xi, g, W, H):
    """Screen-space quantities of Gaussians g in one view: u, v, conic A, B, C, z, opacity, r, g, b, and the
    pixel radius."""
    means, ls, quats, logits, col = (p[g] for p in P)
    fx, fy, cx, cy = cam[:4]
    R0, t0 = cam[4:13].view(3, 3), cam[13:16]
    o = torch.zeros((), dtype=torch.float64, device=DEV)
    S = torch.stack([torch.stack([o, -xi[5], xi[4]]), torch.stack([xi[5], o, -xi[3]]), torch.stack([-xi[4], xi[3], o])])
    R, t = R0 + S @ R0, t0 + S @ t0 + xi[:3]  # Exp(xi) applied on the left, to first order at xi = 0
    pc = means @ R.T + t
    z = pc[:, 2]
    M = _rotation(torch.nn.functional.normalize(quats, dim=1)) * torch.exp(ls)[:, None, :]
    N = R @ M
    limx, limy = 1.3 * 0.5 * W / fx, 1.3 * 0.5 * H / fy
    tx, ty = torch.clamp(pc[:, 0] / z, -limx, limx), torch.clamp(pc[:, 1] / z, -limy, limy)
    m1 = (fx / z)[:, None] * (N[:, 0] - tx[:, None] * N[:, 2])
    m2 = (fy / z)[:, None] * (N[:, 1] - ty[:, None] * N[:, 2])
    a, b, c = (m1 * m1).sum(1) + 0.3, (m1 * m2).sum(1), (m2 * m2).sum(1) + 0.3
    k = torch.linalg.cross(m1, m2)
    det = (k * k).sum(1) + 0.3 * (a + c - 0.6) + 0.09
    if col.dim() == 3:
        d = means + R.T @ t
        col = _sh_colour(col, torch.nn.functional.normalize(d, dim=1))
    s = torch.stack([fx * pc[:, 0] / z + cx, fy * pc[:, 1] / z + cy, c / det, -b / det, a / det, z, torch.sigmoid(logits)], 1)
    lam = 0.5 * (a + c) + torch.sqrt(torch.clamp_min((0.5 * (a - c)) ** 2 + b * b, 0.1))
    return torch.cat([s, col], 1), torch.ceil(3 * torch.sqrt(lam)).detach()


def _lists(vis, rects, W, H, K):
    """Pairs of every tile in depth order: the item of each pair, and each tile's first pair and count."""
    Tx, Ty = (W + 15) // 16, (H + 15) // 16
    cnt = (rects[:, 1] - rects[:, 0]) * (rects[:, 3] - rects[:, 2])
    order = torch.sort(vis["z"].float(), stable=True).indices
    item = torch.repeat_interleave(order, cnt[order])
    first = torch.cumsum(cnt[order], 0) - cnt[order]
    j = torch.arange(item.numel(), device=DEV) - torch.repeat_interleave(first, cnt[order])
    w = (rects[:, 1] - rects[:, 0])[item]
    tile = vis["k"][item] * (Tx * Ty) + (rects[item, 2] + j // w) * Tx + rects[item, 0] + j % w
    tile, o = torch.sort(tile, stable=True)
    n = torch.bincount(tile, minlength=K * Tx * Ty)
    return item[o], torch.cumsum(n, 0) - n, n


def _composite(S, item, start, count, c, upstream, want):
    """Images [K, 5, H, W] (rgb, depth, T) and, with `want`, the gradient of the items' screen quantities for
    upstream(images of a batch of tiles, view, pixel rows, pixel columns) -> gradient of those images."""
    W, H, K = c["W"], c["H"], c["K"]
    Tx, Ty = (W + 15) // 16, (H + 15) // 16
    img = torch.zeros((5, K * H * W), dtype=torch.float64, device=DEV)
    img[4] = 1
    dS = torch.zeros_like(S) if want else None
    tiles = torch.argsort(count, descending=True)
    tiles = tiles[count[tiles] > 0]
    lens = count[tiles].cpu()
    q = torch.arange(256, device=DEV)
    i = 0
    pad = torch.cat([S, torch.zeros_like(S[:1])])  # opacity 0
    while i < len(tiles):
        L = int(lens[i])
        b = tiles[i:i + max(1, 48_000_000 // (256 * L))]
        i += len(b)
        j = torch.arange(L, device=DEV)
        on = j < count[b][:, None]
        ids = torch.where(on, item[torch.where(on, start[b][:, None] + j, 0)], S.shape[0])
        k, tt = b // (Tx * Ty), b % (Tx * Ty)
        py, px = (tt // Tx * 16)[:, None] + q // 16, (tt % Tx * 16)[:, None] + q % 16
        s = pad[ids].requires_grad_(want)
        with torch.set_grad_enabled(want):
            dx = s[:, :, 0, None] - (px + 0.5)[:, None].double()
            dy = s[:, :, 1, None] - (py + 0.5)[:, None].double()
            p = -0.5 * (s[:, :, 2, None] * dx * dx + 2 * s[:, :, 3, None] * dx * dy + s[:, :, 4, None] * dy * dy)
            raw = s[:, :, 6, None] * torch.exp(p)
            alpha = torch.where(raw > 0.99, 0.99, raw)
            with torch.no_grad():
                keep = (p <= 0) & (alpha >= 1 / 255)
                keep &= torch.cumprod(1 - torch.where(keep, alpha, 0), 1) >= 1e-4
            alpha = torch.where(keep, alpha, 0)
            T = torch.cumprod(1 - alpha, 1)
            w = alpha * torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
            out = torch.cat([torch.einsum("blp,blc->bcp", w, s[:, :, [7, 8, 9, 5]]), T[:, -1:]], 1)
        ok = (px < W) & (py < H)
        at = (k[:, None] * H + py) * W + px
        img[:, at[ok]] = out.detach().transpose(0, 1)[:, ok]
        if want:
            g = upstream(out.detach(), torch.where(ok, at, 0)) * ok[:, None]
            ds, = torch.autograd.grad(out, s, g)
            dS.index_add_(0, ids[on], ds[on])
            del ds
        del dx, dy, p, raw, alpha, T, w, out, s
    return img.view(5, K, H, W), dS


def _render64(c, P, cams, upstream=None):
    """(images, gradients of P and of the poses) in 64 bits."""
    W, H, K = c["W"], c["H"], c["K"]
    Tx, Ty = (W + 15) // 16, (H + 15) // 16
    zero = torch.zeros((K, 6), dtype=torch.float64, device=DEV)
    cams = cams.double()
    gs, ks, Ss, rects = [], [], [], []
    for k in range(K):
        z = P[0] @ cams[k, 10:13] + cams[k, 15]
        g = torch.nonzero(z > NEAR)[:, 0]
        s, r = _project(P, cams[k], zero[k], g, W, H)
        lim = lambda v, n: torch.clamp(torch.floor(v), 0, n).long()  # noqa: E731
        rect = torch.stack([lim((s[:, 0] - r) / 16, Tx), lim((s[:, 0] + r) / 16 + 1, Tx),
                            lim((s[:, 1] - r) / 16, Ty), lim((s[:, 1] + r) / 16 + 1, Ty)], 1)
        on = ((rect[:, 1] > rect[:, 0]) & (rect[:, 3] > rect[:, 2]) & (s[:, 6] >= 1 / 256))
        gs.append(g[on])
        ks.append(torch.full_like(gs[-1], k))
        Ss.append(s[on])
        rects.append(rect[on])
    S = torch.cat(Ss)
    item, start, count = _lists({"z": S[:, 5], "k": torch.cat(ks)}, torch.cat(rects), W, H, K)
    img, dS = _composite(S, item, start, count, c, upstream, upstream is not None)
    if upstream is None:
        return img, None, None
    P = [p.detach().requires_grad_() for p in P]
    xi = zero.clone().requires_grad_()
    total = [torch.zeros_like(p) for p in (*P, xi)]
    at = 0
    for k in range(K):  # one view's projection at a time
        s, _ = _project(P, cams[k], xi[k], gs[k], W, H)
        for t, d in zip(total, torch.autograd.grad(s, (*P, xi), dS[at:at + len(gs[k])])):
            t += d
        at += len(gs[k])
    return img, total[:5], total[5]


def _l1(rgb_t, depth_t, H, W):
    """upstream() of the key-frame loss: mean |R - R*| over 3HW + lambda mean |D - D*| over HW, per view."""
    t = torch.cat([rgb_t.transpose(0, 1).reshape(3, -1), depth_t.reshape(1, -1)]).double()
    w = torch.tensor([1 / (3 * H * W)] * 3 + [LAMBDA / (H * W)], dtype=torch.float64, device=DEV)[:, None]

    def up(out, at):
        g = torch.sign(out[:, :4] - t[:, at].transpose(0, 1)) * w
        return torch.cat([g, torch.zeros_like(out[:, 4:])], 1)

    def value(img):
        return (torch.abs(img[:4].reshape(4, -1) - t) * w).sum().reshape(1)

    return up, value


def exact(case, seed):
    c, op = case, case["op"]
    if op == "sort":
        return None
    if op == "adam":
        masters, grads, state = _adam_inputs(c, seed)
        lr = {"means": 1.6e-4, "log_scales": 5e-3, "quats": 1e-3, "opacity_logits": 5e-2, "rgb": 2.5e-3}
        total = (state.numel() - 1) // 2
        f32 = lambda v: torch.tensor(v, dtype=torch.float32, device=DEV).double()  # noqa: E731  (as the call takes it)
        b1, b2, eps, t = f32(0.9), f32(0.999), f32(1e-15), 201.0
        m, v, off, out = state[:total].double(), state[total:2 * total].double(), 0, []
        ms, vs = [], []
        for k in PARAMS:
            n = masters[k].numel()
            g = grads[k].double().reshape(-1)
            mk = b1 * m[off:off + n] + (1 - b1) * g
            vk = b2 * v[off:off + n] + (1 - b2) * g * g
            step = f32(lr[k]) * (mk / (1 - b1 ** t)) / (torch.sqrt(vk / (1 - b2 ** t)) + eps)
            out.append((masters[k].double().reshape(-1) - step).view(masters[k].shape))
            ms.append(mk)
            vs.append(vk)
            off += n
        return {"masters": out, "storage": out, "m": torch.cat(ms), "v": torch.cat(vs),
                "steps": f32(201.0).reshape(1)}
    if op == "metrics":
        x, y = (i.double() for i in _images(c, seed))
        d = torch.arange(11, dtype=torch.float64, device=DEV) - 5
        w = torch.exp(-d * d / (2 * 1.5 ** 2))
        w = (w / w.sum())
        win = (w[:, None] * w[None, :])[None, None]
        B, C, H, W = x.shape
        blur = lambda i: torch.nn.functional.conv2d(i.reshape(B * C, 1, H, W), win, padding=5).view(B, C, H, W)  # noqa: E731
        mx, my = blur(x), blur(y)
        vx, vy, cxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
        s = ((2 * mx * my + 1e-4) * (2 * cxy + 9e-4)) / ((mx * mx + my * my + 1e-4) * (vx + vy + 9e-4))
        return {"psnr": -10 * torch.log10(((x - y) ** 2).mean((1, 2, 3))), "ssim": s.mean((1, 2, 3)), "map": s}
    P = [p.double() for p in _map_arrays(c, seed)]
    cams = _cameras(c, seed)
    images = lambda img: {"rgb": img[:3].transpose(0, 1), "depth": img[3], "T": img[4], "last": None}  # noqa: E731
    if op == "render":
        return images(_render64(c, P, cams)[0])
    if op == "autograd":
        up = torch.cat([_upstream(c, seed)[0].transpose(0, 1).reshape(3, -1)]
                       + [u.reshape(1, -1) for u in _upstream(c, seed)[1:]]).double()
        img, grads, pose = _render64(c, P, cams, lambda out, at: up[:, at].transpose(0, 1))
        return {"out": [img[:3].transpose(0, 1), img[3], img[4]], "grads": [*grads, pose]}
    if op == "track":
        seen, _, _ = _render64(c, P, cams)
        n_rgb, n_depth = _sensor_noise(c, seed)
        frames, cams = (seen[:3].transpose(0, 1) + n_rgb, seen[3] + n_depth), _off_pose(cams, seed)
    else:
        frames = _frames(c, seed)
    up, value = _l1(*frames, c["H"], c["W"])
    img, grads, pose = _render64(c, P, cams, up)
    if op == "track":  # the first step of Adam from zero moments moves every component by its rate
        return {"cams": None, "pose_grad": pose, "loss": value(img)}
    return {"grads": dict(zip((*PARAMS, "pose"), (*grads, pose))), "loss": value(img), **images(img)}
