"""What a user of this framework has it do, as cases that can be timed.

A case is a dict of plain values.  listed() gives the fixed ones, draw() further
ones of the same ranges; prepare() builds what a program has in hand before the
call (a loaded scene, a camera, output buffers), run() is one pass through the
public entry points of paper_2310_08528_gb300.fs4d, work() the bytes and operations
the path cannot do without, exact() the same outputs in 64 bits from plain torch.

Scenes follow the shapes of scenegen (tiny, object, room, stress), drawn with
torch on the GPU so that a case is prepared quickly, with wider MLP weights so that
the deformation is visible.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2310_08528_gb300 import fs4d, scenegen

TILE = 16
MLP_STD = 0.08
PREC = {"fp32": fs4d.FP32, "bf16": fs4d.BF16}

# Scene shapes: HexPlane levels and time resolution, features, SH degree, mean
# log-scale, whether the means fill a room (else a ball).
SCENES = {
    "tiny": dict(res=(32,), rt=8, h=16, sh=0, scale=-4.0, room=False),
    "object": dict(res=(64, 128), rt=25, h=32, sh=3, scale=-4.0, room=False),
    "room": dict(res=(64, 128), rt=150, h=32, sh=3, scale=-3.5, room=True),
    "stress": dict(res=(64, 128, 256), rt=300, h=32, sh=3, scale=-2.5, room=False),
}


def listed():
    return [
        # the smallest frame a viewer or a test asks for: the host path and the launches count
        {"name": "frame_tiny_fp32", "do": "frame", "scene": "tiny", "n": 2000, "width": 128, "height": 128,
         "prec": "fp32", "heads": False},
        # the framework's default precision on a real-scene-sized frame
        {"name": "frame_room_fp32", "do": "frame", "scene": "room", "n": 300_000, "width": 1352, "height": 1014,
         "prec": "fp32", "heads": False},
        # the headline workload, queued without a host synchronisation as a real-time loop does
        {"name": "frame_object_bf16_async", "do": "async", "scene": "object", "n": 100_000, "width": 800, "height": 800,
         "prec": "bf16", "heads": False},
        # the same object with the colour and opacity heads
        {"name": "frame_object_bf16_heads", "do": "frame", "scene": "object", "n": 100_000, "width": 800, "height": 800,
         "prec": "bf16", "heads": True},
        # the largest frame: 2M large Gaussians at 1080p (more than a billion tile pairs)
        {"name": "frame_stress_bf16", "do": "frame", "scene": "stress", "n": 2_000_000, "width": 1920, "height": 1080,
         "prec": "bf16", "heads": False},
        # tracking: the trajectories of every Gaussian over 16 timestamps in one call
        {"name": "deform_track_bf16", "do": "deform", "scene": "object", "n": 100_000, "steps": 16, "prec": "bf16"},
        # one deformation in the default precision
        {"name": "deform_room_fp32", "do": "deform", "scene": "room", "n": 300_000, "steps": 1, "prec": "fp32"},
        # the stages as calls of their own: projection with SH colour, binning, compositing
        {"name": "project_room", "do": "project", "scene": "room", "n": 300_000, "width": 1352, "height": 1014},
        {"name": "bin_sort_object", "do": "bin_sort", "scene": "object", "n": 100_000, "width": 800, "height": 800},
        {"name": "composite_object", "do": "composite", "scene": "object", "n": 100_000, "width": 800, "height": 800},
        # the gradients of one view into every parameter group (a custom training loop)
        {"name": "backward_object_fp32", "do": "backward", "scene": "object", "n": 100_000, "width": 800, "height": 800,
         "prec": "fp32"},
        # the on-device training step at the size a real scene is trained at
        {"name": "train_room_bf16", "do": "train", "scene": "room", "n": 300_000, "width": 1352, "height": 1014,
         "prec": "bf16"},
    ]


def draw(rng):
    """One more case: the same calls over the range of sizes, odd and ragged ones among them."""
    do = rng.choice(["frame", "frame", "async", "deform", "deform", "project", "bin_sort", "composite", "backward",
                     "train"])
    scene = rng.choice(["tiny", "object", "object", "room", "stress"] if do in ("frame", "deform", "project")
                       else ["tiny", "object", "object", "room"])
    top = {"tiny": 20_000, "object": 300_000, "room": 300_000, "stress": 1_000_000}[scene]
    n = int(round(math.exp(rng.uniform(math.log(1000), math.log(top)))))
    case = {"do": do, "scene": scene, "n": n}
    if do == "deform":
        case["steps"] = rng.choice([1, 1, 2, 5, 16])
    else:
        case["width"] = int(round(math.exp(rng.uniform(math.log(100), math.log(1920)))))
        case["height"] = max(64, min(1080, int(round(case["width"] * rng.uniform(0.5, 1.1)))))
    if do not in ("project", "bin_sort", "composite"):
        case["prec"] = rng.choice(["fp32", "bf16"])
    if do in ("frame", "async"):
        case["heads"] = scene in ("object", "room") and rng.random() < 0.25
    return case


# ----------------------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _mixture(g, n, room):
    """Means of a Gaussian mixture inside the unit ball, or inside the 6x4x6 box of a room."""
    box = torch.tensor([3.0, 2.0, 3.0] if room else [1.0, 1.0, 1.0], device="cuda")
    k, std = (64, 0.35) if room else (32, 0.15)
    centres = torch.rand(4 * k, 3, generator=g, device="cuda") * 2 - 1
    centres = (centres if room else 0.7 * centres[centres.norm(dim=1) <= 1])[:k] * box
    got, have = [], 0
    while have < n:
        at = torch.randint(0, centres.shape[0], (2 * n,), generator=g, device="cuda")
        p = centres[at] + std * torch.randn(2 * n, 3, generator=g, device="cuda")
        p = p[(p.abs() <= box).all(1)] if room else p[p.norm(dim=1) <= 1]
        got.append(p)
        have += p.shape[0]
    return torch.cat(got)[:n].contiguous(), box


def _scene(case, seed):
    """A scene of the case's shape as float32 CUDA tensors, and what describes its grid."""
    s, n, g = SCENES[case["scene"]], case["n"], _generator(seed)

    def normal(mean, std, *shape):
        return mean + std * torch.randn(*shape, generator=g, device="cuda")

    p = {}
    if case["scene"] == "tiny":
        p["means"], box = torch.rand(n, 3, generator=g, device="cuda") * 2 - 1, torch.ones(3, device="cuda")
    else:
        p["means"], box = _mixture(g, n, s["room"])
    p["log_scales"] = normal(s["scale"], 0.5, n, 3)
    p["quats"] = torch.nn.functional.normalize(normal(0, 1, n, 4), dim=1)
    p["opacity_logits"] = normal(0, 1, n)
    p["sh"] = normal(0, 0.05, n, (s["sh"] + 1) ** 2, 3)
    p["sh"][:, 0] = (torch.rand(n, 3, generator=g, device="cuda") - 0.5) / 0.28209479177387814
    cells = sum(a * b for a, b, _ in scenegen.plane_shapes(s["res"], s["rt"], 1))
    p["planes"] = normal(1.0, 0.1, cells * s["h"])
    parts = []
    heads = (s["sh"] + 1) ** 2 if case.get("heads") else 0
    for k, (o, i) in enumerate(scenegen.mlp_layer_shapes(s["h"] * len(s["res"]), 64, heads)):
        parts += [normal(0, MLP_STD if k < 8 else 0.05, o * i), normal(0, 0.02, o)]
    p["mlp"] = torch.cat(parts)
    return {k: v.contiguous() for k, v in p.items()}, box


def _host_scene(case, p, box):
    s, host = SCENES[case["scene"]], {k: v.cpu().numpy() for k, v in p.items()}
    lim = [float(v) for v in box.cpu()]
    return scenegen.Scene(host["means"], host["log_scales"], host["quats"], host["opacity_logits"], host["sh"],
                          s["sh"], tuple(-v for v in lim), tuple(lim), s["res"], s["rt"], s["h"], host["planes"], 64,
                          host["mlp"], bool(case.get("heads")))


def _view(case, seed):
    """A camera of the scene's kind and a timestamp."""
    rng = np.random.default_rng(int(seed))
    w, h = case["width"], case["height"]
    if SCENES[case["scene"]]["room"]:
        cam = scenegen.forward_cameras(1, w, h, seed=int(rng.integers(1 << 30)))[0]
    else:
        cam = scenegen.hemisphere_cameras(50, width=w, height=h, seed=int(rng.integers(1 << 30)))[int(rng.integers(50))]
    return cam, float(rng.uniform())


def prepare(case, seed):
    do = case["do"]
    p, box = _scene(case, seed)
    st = {"do": do, "prec": PREC[case.get("prec", "fp32")]}
    if "width" in case:
        st["cam"], st["t"] = _view(case, seed)
    if do in ("project", "bin_sort", "composite"):
        st["ctx"] = fs4d.Context(0)
        if do == "project":
            st["args"] = (p["means"], p["quats"], p["log_scales"], p["opacity_logits"], p["sh"],
                          SCENES[case["scene"]]["sh"], st["cam"])
            return st
        tx, ty = _tiles(st["cam"])
        q = _stage_inputs(case, p, st["cam"])
        if do == "bin_sort":
            rect = _even_rects(case, q["xy"], st["cam"], seed)
            st["args"] = (q["depth"], rect, tx, ty, int(_pair_count(rect)))
        else:
            st["args"] = (case["width"], case["height"], q["ranges"], q["values"], q["xy"], q["conic_opacity"],
                          q["rgb"])
        return st

    ctx = st["ctx"] = fs4d.Context(0)
    scene = _host_scene(case, p, box)
    if do == "train":  # the target is a frame of the same scene with slightly different planes
        other = ctx.load_scene(scenegen.perturb_planes(scene, int(seed) % 10_000))
        st["target"] = ctx.render(other, st["cam"], st["t"], fs4d.FP32)
        ctx.unload_scene(other)
    sid = st["sid"] = ctx.load_scene(scene)
    if do == "deform":
        rng = np.random.default_rng(int(seed))
        st["ts"] = np.sort(rng.uniform(size=case["steps"])).astype(np.float32)
        t, n = case["steps"], case["n"]
        st["out"] = tuple(torch.empty(t, n, k, device="cuda") for k in (3, 4, 3))
    elif do in ("frame", "async"):
        st["image"] = torch.empty(case["height"], case["width"], 3, device="cuda")
        ctx.render(sid, st["cam"], st["t"], st["prec"], image=st["image"])
        if do == "async":  # sized with room to spare, as a loop over many views does
            ctx.reserve(sid, case["width"], case["height"], 2 * ctx.last_pairs() + 4096)
            raw = np.frombuffer(bytes(fs4d.camera_struct(st["cam"])), np.float32).copy()
            st["d_cam"] = torch.from_numpy(raw).cuda()
            st["d_t"] = torch.tensor([st["t"]], device="cuda")
    elif do == "backward":
        g = _generator(seed + 1)
        st["dl"] = torch.randn(case["height"], case["width"], 3, generator=g, device="cuda") / case["width"]
        st["shapes"] = {k: v.shape for k, v in p.items()}
    elif do == "train":
        st["trainer"] = fs4d.Trainer(ctx, sid, 3000)
        st["losses"] = torch.zeros(2, device="cuda")
        st["params"] = {k: torch.empty_like(v) for k, v in p.items()}
    return st


def run(st):
    ctx, do = st["ctx"], st["do"]
    if do == "frame":
        return ctx.render(st["sid"], st["cam"], st["t"], st["prec"], image=st["image"])
    if do == "async":
        ctx.render_async(st["sid"], st["cam"], st["d_cam"], st["d_t"], st["image"], st["prec"])
        return st["image"]
    if do == "deform":
        return ctx.deform(st["sid"], st["ts"], st["prec"], out=st["out"])
    if do == "project":
        return ctx.project(*st["args"])
    if do == "bin_sort":
        return ctx.bin_sort(*st["args"])
    if do == "composite":
        return ctx.composite(*st["args"])
    if do == "backward":
        image, frame = ctx.render_saved(st["sid"], st["cam"], st["t"], st["prec"])
        grads = {k: torch.zeros(s, device="cuda") for k, s in st["shapes"].items()}
        ctx.render_backward(frame, st["dl"], grads)
        ctx.frame_free(frame)
        return {"image": image, **grads}
    st["trainer"].step(st["cam"], st["t"], st["target"], st["prec"], losses=st["losses"])
    out = fs4d.Grads(**{k: int(v.data_ptr()) for k, v in st["params"].items()})
    ctx.call("fs4d_read_scene", st["sid"], ctypes.byref(out), 1)
    return {"losses": st["losses"], **st["params"]}


def work(case):
    s, n, do = SCENES[case["scene"]], case["n"], case["do"]
    k3, pix = 3 * (s["sh"] + 1) ** 2, case.get("width", 0) * case.get("height", 0)
    hl = s["h"] * len(s["res"])
    mlp = 2 * (hl * 64 + 4 * 64 * 64 + 64 * 10) + 6 * 8 * hl        # operations of one deformation
    esize = 2 if case.get("prec") == "bf16" else 4
    shapes = scenegen.plane_shapes(s["res"], s["rt"], s["h"])       # spatial planes whole, two rows of the time planes
    rows = sum((rb if i % 6 < 3 else min(rb, 2)) * ra * h for i, (rb, ra, h) in enumerate(shapes))
    color = 2 * (64 * 64 * 2 + 64 * (k3 + 1)) if case.get("heads") else 0
    deform = {"bytes": n * 40 + rows * esize, "flops": n * mlp}
    project = {"bytes": n * (40 + 4 + 4 * k3 + 56), "flops": n * (300 + 4 * k3)}
    if do == "deform":
        t = case["steps"]
        return {"bytes": n * 40 * (1 + t) + rows * esize, "flops": n * t * mlp}
    if do == "project":
        return project
    if do == "bin_sort":   # about eleven tile pairs a Gaussian: key and value written once
        return {"bytes": n * (20 + 11 * 12), "flops": n * 11}
    if do == "composite":  # each pixel blends some tens of terms
        return {"bytes": n * (36 + 11 * 4) + pix * 20, "flops": pix * 60 * 15}
    frame = {"bytes": deform["bytes"] + n * (4 + 4 * k3) + pix * 12,
             "flops": deform["flops"] + project["flops"] + n * color + pix * 60 * 15}
    if do in ("frame", "async"):
        return frame
    params = n * (11 + k3) + sum(a * b * h for a, b, h in shapes)
    back = {"bytes": 2 * frame["bytes"] + 4 * params + pix * 12, "flops": 3 * frame["flops"]}
    if do == "backward":
        return back
    return {"bytes": back["bytes"] + 4 * 6 * params + 12 * pix, "flops": back["flops"] + 12 * params}


# ----------------------------------------------------------------------------- the same in 64 bits

def _tiles(cam):
    return (cam.width + TILE - 1) // TILE, (cam.height + TILE - 1) // TILE


def _pair_count(rect):
    r = rect.long()
    return ((r[:, 2] - r[:, 0]) * (r[:, 3] - r[:, 1])).sum()


def _deform64(case, p, box, t):
    """(means, quats, log_scales) at time t, and the features that the heads read."""
    s, x = SCENES[case["scene"]], p["means"]
    u = torch.cat([x / box, torch.full_like(x[:, :1], 2 * t - 1)], 1).clamp(-1, 1)
    at, feats, prod = 0, [], None
    for i, (rb, ra, h) in enumerate(scenegen.plane_shapes(s["res"], s["rt"], s["h"])):
        a, b = scenegen.PLANE_AXES[i % 6]
        plane = p["planes"][at:at + ra * rb * h].view(rb * ra, h)
        at += ra * rb * h
        ga, gb = (u[:, a] + 1) / 2 * (ra - 1), (u[:, b] + 1) / 2 * (rb - 1)
        ia, ib = ga.detach().floor().clamp(0, ra - 2).long(), gb.detach().floor().clamp(0, rb - 2).long()
        fa, fb = (ga - ia)[:, None], (gb - ib)[:, None]
        v = ib * ra + ia
        val = (1 - fa) * (1 - fb) * plane[v] + fa * (1 - fb) * plane[v + 1] \
            + (1 - fa) * fb * plane[v + ra] + fa * fb * plane[v + ra + 1]
        prod = val if i % 6 == 0 else prod * val
        if i % 6 == 5:
            feats.append(prod)
    heads = (s["sh"] + 1) ** 2 if case.get("heads") else 0
    layers, at = [], 0
    for o, i in scenegen.mlp_layer_shapes(s["h"] * len(s["res"]), 64, heads):
        layers.append((p["mlp"][at:at + o * i].view(o, i), p["mlp"][at + o * i:at + o * i + o]))
        at += o * i + o

    def lin(k, v):
        return v @ layers[k][0].T + layers[k][1]

    fd = torch.relu(lin(1, torch.relu(lin(0, torch.cat(feats, 1)))))
    out = [lin(k + 1, torch.relu(lin(k, fd))) for k in range(2, len(layers), 2)]
    q = dict(p, means=x + out[0], quats=p["quats"] + out[1], log_scales=p["log_scales"] + out[2])
    if heads:
        q["sh"] = p["sh"] + out[3].view(p["sh"].shape)
        q["opacity_logits"] = p["opacity_logits"] + out[4][:, 0]
    return q


def _basis(deg, d):
    x, y, z = d.unbind(1)
    out = [torch.full_like(x, math.sqrt(1 / (4 * math.pi)))]
    if deg > 0:
        c = math.sqrt(3 / (4 * math.pi))
        out += [c * y, c * z, c * x]
    if deg > 1:
        c = math.sqrt(15 / math.pi)
        out += [c / 2 * x * y, c / 2 * y * z, math.sqrt(5 / math.pi) / 4 * (3 * z * z - 1), c / 2 * x * z,
                c / 4 * (x * x - y * y)]
    if deg > 2:
        a, b, c = math.sqrt(35 / (2 * math.pi)) / 4, math.sqrt(105 / math.pi) / 2, math.sqrt(21 / (2 * math.pi)) / 4
        out += [a * y * (3 * x * x - y * y), b * x * y * z, c * y * (5 * z * z - 1),
                math.sqrt(7 / math.pi) / 4 * z * (5 * z * z - 3), c * x * (5 * z * z - 1), b / 2 * z * (x * x - y * y),
                a * x * (x * x - 3 * y * y)]
    return torch.stack(out, 1)


def _project64(case, q, cam):
    """xy, conic and opacity, colour, depth and tile rectangle of every Gaussian (zeros where it is not seen)."""
    s, m = SCENES[case["scene"]], torch.tensor(cam.world_to_cam.astype(np.float64), device="cuda")
    fx, fy, cx, cy, near = (float(np.float32(v)) for v in (cam.fx, cam.fy, cam.cx, cam.cy, cam.znear))
    x = q["means"]
    pc = x @ m[:3, :3].T + m[:3, 3]
    depth = pc[:, 2]
    ahead = depth > near
    z = torch.where(ahead, depth, torch.ones_like(depth))
    w, i, j, k = torch.nn.functional.normalize(q["quats"], dim=1).unbind(1)
    rot = torch.stack([1 - 2 * (j * j + k * k), 2 * (i * j - w * k), 2 * (i * k + w * j),
                       2 * (i * j + w * k), 1 - 2 * (i * i + k * k), 2 * (j * k - w * i),
                       2 * (i * k - w * j), 2 * (j * k + w * i), 1 - 2 * (i * i + j * j)], 1).view(-1, 3, 3)
    lx, ly = 1.3 * cam.width / (2 * fx), 1.3 * cam.height / (2 * fy)
    rx, ry = (pc[:, 0] / z).clamp(-lx, lx), (pc[:, 1] / z).clamp(-ly, ly)
    o = torch.zeros_like(z)
    jac = torch.stack([fx / z, o, -fx * rx / z, o, fy / z, -fy * ry / z], 1).view(-1, 2, 3)
    a = jac @ m[:3, :3] @ rot * torch.exp(q["log_scales"])[:, None, :]
    cov = a @ a.transpose(1, 2)
    ca, cb, cc = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = ca * cc - cb * cb
    u = torch.stack([fx * pc[:, 0] / z + cx, fy * pc[:, 1] / z + cy], 1)
    with torch.no_grad():
        rad = torch.ceil(3 * torch.sqrt(0.5 * (ca + cc) + torch.sqrt((0.5 * (ca - cc)) ** 2 + cb * cb)))
        lim = torch.tensor(_tiles(cam), device="cuda")
        lo = torch.minimum(torch.floor((u - rad[:, None]) / TILE).long().clamp(min=0), lim)
        hi = torch.minimum((torch.floor((u + rad[:, None]) / TILE).long() + 1).clamp(min=0), lim)
        seen = ahead & (det > 0) & (hi > lo).all(1)
        rect = torch.cat([lo, hi], 1) * seen[:, None]
    d = torch.nn.functional.normalize(x + m[:3, :3].T @ m[:3, 3], dim=1)
    rgb = torch.relu(torch.einsum("nk,nkc->nc", _basis(s["sh"], d), q["sh"]) + 0.5)
    conic = torch.stack([cc / det, -cb / det, ca / det], 1)
    see = seen[:, None]
    return {"xy": torch.where(see, u, torch.zeros_like(u)),
            "conic_opacity": torch.cat([torch.where(see, conic, torch.zeros_like(conic)),
                                        torch.sigmoid(q["opacity_logits"])[:, None]], 1),
            "rgb": torch.where(see, rgb, torch.zeros_like(rgb)), "depth": depth, "rect": rect.int()}


def _lists(rect, depth, tx, ty):
    """Per-tile Gaussian lists in (depth, index) order: values, and [start, end) of each tile."""
    r = rect.long()
    w, cnt = r[:, 2] - r[:, 0], (r[:, 2] - r[:, 0]) * (r[:, 3] - r[:, 1])
    order = torch.sort(depth.float(), stable=True)[1]
    g = torch.repeat_interleave(order, cnt[order])
    start = torch.cumsum(cnt[order], 0) - cnt[order]
    k = torch.arange(g.numel(), device="cuda") - torch.repeat_interleave(start, cnt[order])
    tile = (r[g, 1] + k // w[g]) * tx + r[g, 0] + k % w[g]
    tile, at = torch.sort(tile, stable=True)
    edge = torch.searchsorted(tile, torch.arange(tx * ty + 1, device="cuda"))
    ranges = torch.stack([edge[:-1], edge[1:]], 1)
    ranges = torch.where((ranges[:, 1] > ranges[:, 0])[:, None], ranges, torch.zeros_like(ranges))
    return g[at].int().contiguous(), ranges.int().contiguous()


def _stage_inputs(case, p, cam):
    """The projection's outputs as a program that calls the later stages has them, in float32."""
    q = _project64(case, {k: v.double() for k, v in p.items()}, cam)
    out = {k: (v if k == "rect" else v.float()).contiguous() for k, v in q.items()}
    if case["do"] == "composite":
        out["values"], out["ranges"] = _lists(out["rect"], out["depth"], *_tiles(cam))
    return out


def _even_rects(case, xy, cam, seed):
    """Tile rectangles around the projected means, their sides the quantiles of the scene's projected sizes in an
    order of the seed's, so that every seed has as many pairs as the next."""
    n, (tx, ty) = case["n"], _tiles(cam)
    z = math.sqrt(2) * torch.erfinv((torch.arange(n, device="cuda") * 2 + 1.0) / n - 1)
    px = cam.fx / (5.5 if SCENES[case["scene"]]["room"] else 4.0) * torch.exp(SCENES[case["scene"]]["scale"] + 0.5 * z)
    side = 1 + torch.floor((6 * px + TILE / 2) / TILE).long()
    w, h = side.clamp(max=tx), side.roll(n // 3).clamp(max=ty)
    at = torch.randperm(n, generator=_generator(seed + 2), device="cuda")
    w, h = w[at], h[at]
    x = torch.minimum(torch.floor(xy[:, 0] / TILE - w / 2 + 0.5).long().clamp(min=0), tx - w)
    y = torch.minimum(torch.floor(xy[:, 1] / TILE - h / 2 + 0.5).long().clamp(min=0), ty - h)
    return torch.stack([x, y, x + w, y + h], 1).int().contiguous()


def _composite64(cam, values, ranges, xy, conic, rgb, dl=None):
    """Image and transmittance; with dl the gradients of sum(dl * image) in place of the transmittance."""
    tx, ty = _tiles(cam)
    image = torch.zeros(ty * TILE, tx * TILE, 3, dtype=torch.float64, device="cuda")
    trans = torch.ones(ty * TILE, tx * TILE, dtype=torch.float64, device="cuda")
    grads = [torch.zeros_like(v) for v in (xy, conic, rgb)]
    dpad = torch.zeros_like(image)
    if dl is not None:
        dpad[:cam.height, :cam.width] = dl
    px = torch.arange(TILE, device="cuda", dtype=torch.float64) + 0.5
    values = values.long()
    for tile, (a, b) in enumerate(ranges.cpu().tolist()):
        if b <= a:
            continue
        x0, y0 = tile % tx * TILE, tile // tx * TILE
        g = values[a:b]
        leaf = [v[g] for v in (xy, conic, rgb)]
        if dl is not None:
            leaf = [v.detach().requires_grad_() for v in leaf]
        with torch.set_grad_enabled(dl is not None):
            dx = (leaf[0][:, 0, None] - (x0 + px))[:, None, :]
            dy = (leaf[0][:, 1, None] - (y0 + px))[:, :, None]
            c = leaf[1][:, :, None, None]
            al = (c[:, 3] * torch.exp(-0.5 * (c[:, 0] * dx * dx + 2 * c[:, 1] * dx * dy + c[:, 2] * dy * dy)))
            al = al.clamp(max=0.99)
            al = torch.where(al.detach() < 1 / 255, torch.zeros_like(al), al).flatten(1)
            t1 = torch.cumprod(1 - al, 0)
            live = t1.detach() >= 1e-4
            t0 = torch.cat([torch.ones_like(t1[:1]), t1[:-1]])
            out = ((al * t0 * live).T @ leaf[2]).view(TILE, TILE, 3)
        box = (slice(y0, y0 + TILE), slice(x0, x0 + TILE))
        image[box] = out.detach()
        trans[box] = torch.where(live, t1.detach(), torch.ones_like(t1)).amin(0).view(TILE, TILE)
        if dl is not None:
            for acc, v in zip(grads, torch.autograd.grad((out * dpad[box]).sum(), leaf)):
                acc.index_add_(0, g, v)
    image = image[:cam.height, :cam.width]
    return (image, grads) if dl is not None else (image, trans[:cam.height, :cam.width])


def exact(case, seed):
    do = case["do"]
    if do in ("train", "bin_sort"):      # Adam's first steps take the sign of a gradient; whole numbers
        return None
    if "width" in case and do != "project" and (case["n"] > 150_000 or case["width"] * case["height"] > 1_000_000
                                                or case["scene"] == "stress"):
        return None                      # too long in 64 bits
    p, box = _scene(case, seed)
    p, box = {k: v.double() for k, v in p.items()}, box.double()
    if do == "deform":
        ts = np.sort(np.random.default_rng(int(seed)).uniform(size=case["steps"])).astype(np.float32)
        qs = [_deform64(case, p, box, float(t)) for t in ts]
        return tuple(torch.stack([q[k] for q in qs]) for k in ("means", "quats", "log_scales"))
    cam, t = _view(case, seed)
    if do == "project":
        q = _project64(case, p, cam)
        return dict(q, radius=None, rect=None)
    if do == "composite":
        q = _stage_inputs(case, {k: v.float() for k, v in p.items()}, cam)
        image, trans = _composite64(cam, q["values"], q["ranges"], *(q[k].double() for k in ("xy", "conic_opacity",
                                                                                            "rgb")))
        return image, trans, None
    t = float(np.float32(t))
    tx, ty = _tiles(cam)
    if do != "backward":
        q = _project64(case, _deform64(case, p, box, t), cam)
        values, ranges = _lists(q["rect"], q["depth"], tx, ty)
        return _composite64(cam, values, ranges, q["xy"], q["conic_opacity"], q["rgb"])[0]
    if case["prec"] != "fp32":           # the gradients of a BF16 frame are those of its float32 deformation
        return None
    dl = torch.randn(case["height"], case["width"], 3, generator=_generator(seed + 1), device="cuda") / case["width"]
    p = {k: v.requires_grad_() for k, v in p.items()}
    q = _project64(case, _deform64(case, p, box, t), cam)
    values, ranges = _lists(q["rect"], q["depth"].detach(), tx, ty)
    three = [q[k] for k in ("xy", "conic_opacity", "rgb")]
    image, grads = _composite64(cam, values, ranges, *(v.detach() for v in three), dl=dl.double())
    torch.autograd.backward(three, grads)
    return {"image": image, **{k: v.grad for k, v in p.items()}}
