"""The work that users of this library have it do, as measurable cases.

Each case is one call, or the few calls that always go together, through the
public Python entry points (`dags.Context` and `autograd`): the mapping and
tracking halves of the SLAM loop, the motion-probability (MP) update, the
learned MP proposal, and the checks between keyframes. Sizes are those of the
repository's own workloads: the 2,000-Gaussian 160x120 scene, the 300,000-
Gaussian 640x480 tracking frame, the 200,000-Gaussian window of 8 keyframes and
the 1,000,000-Gaussian 1200x680 full loop.

Scenes are made on the GPU from the seed: Gaussians on the surfaces of the
6 x 6 x 3 m room and its ellipsoids (`synth`'s room, sampled here with torch),
and RGB-D frames ray-cast from the same analytic scene.

`exact` is the same mathematics in plain 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_2602_21644_gb300 import autograd, dags, synth

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
TILE = 16
ALPHA_MIN, ALPHA_MAX, T_MIN, DILATION, Z_NEAR, GUARD = 1 / 255, 0.99, 1e-4, 0.3, 0.2, 1.3
FPS = 30.0


# --------------------------------------------------------------------- cases

def listed():
    return [
        # The smallest scene, where launches and host work count: an interactive
        # preview, a unit of a test suite.
        dict(name="splat_tiny", kind="splat", n=2000, width=160, height=120, scene="box", autograd=True),
        # One frame's loss with the gradients of the map and the pose, as an
        # optimiser that keeps its buffers calls it.
        dict(name="splat_frame", kind="splat", n=300_000, width=640, height=480, scene="room", autograd=False),
        # Rendered channels for a caller's own loss, at sizes that divide nothing.
        dict(name="render_ragged", kind="render", n=100_003, width=637, height=477, scene="room"),
        # One mapping iteration over the keyframe window: render, adjoint, the
        # motion-consistency term and the Adam step on the map.
        dict(name="mapping_window", kind="mapping", n=200_000, width=640, height=480, views=8),
        # The same at the scale of the full loop: the largest splatting call.
        dict(name="mapping_full", kind="mapping", n=1_000_000, width=1200, height=680, views=8),
        # First-order tracking of a few frames, each 100 pose iterations from the
        # previous frame's pose.
        dict(name="track_frames", kind="track", n=300_000, width=640, height=480, frames=4, iters=100),
        # A frame's second-order tracking: 15 Levenberg-Marquardt iterations.
        dict(name="track_lm", kind="lm", n=300_000, width=640, height=480, iters=15),
        # A frame's MP update and the decision whether to refresh the instance
        # prior, on a frame with a fresh prior.
        dict(name="mp_update", kind="mp", n=300_000, width=640, height=480, scales=1, learned=False, fresh=True),
        # A frame between two refreshes at full scale: the network proposes the
        # per-pixel MP of one frame and the update associates it over a pyramid.
        dict(name="mp_learned_frame", kind="mp", n=1_000_000, width=1200, height=680, scales=3, learned=True,
             fresh=False),
        # Batched inference of the MP network, as offline evaluation runs it.
        dict(name="net_infer", kind="infer", batch=16, width=640, height=480),
        # One training step of the MP network.
        dict(name="net_train", kind="train", batch=16, width=640, height=480),
        # The checks when a keyframe is taken: epipolar verification of the
        # matches and the edge-warp term between the two frames.
        dict(name="keyframe_checks", kind="keyframe", n=300_000, width=640, height=480, matched=20_000, per_gauss=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _image(rng, lo, hi):
    """A frame of lo to hi pixels across, 4:3 to 16:9, odd sizes among them."""
    w = _log(rng, lo, hi)
    return w, max(90, int(w * rng.uniform(0.56, 0.75)))


def draw(rng):
    kind = rng.choice(["splat", "splat", "render", "mapping", "mapping", "track", "lm", "mp", "mp", "infer", "train",
                       "keyframe"])
    if kind in ("infer", "train"):
        w, h = _image(rng, 160, 640)
        return dict(kind=kind, batch=_log(rng, 1, 16), width=w, height=h)
    big = kind in ("splat", "render", "mapping", "mp")
    w, h = _image(rng, 160, 1200 if big else 640)
    h = min(h, 680 if big else 480)
    n = min(1_000_000 if big else 300_000, max(2000, int(w * h * math.exp(rng.uniform(math.log(0.1), math.log(1.25))))))
    case = dict(kind=kind, n=n, width=w, height=h)
    if kind in ("splat", "render"):
        case["scene"] = rng.choice(["room", "room", "room", "box"]) if n <= 20_000 else "room"
        if kind == "splat":
            case["autograd"] = rng.random() < 0.5
    elif kind == "mapping":
        case["views"] = rng.randint(2, 8)
    elif kind == "track":
        case.update(frames=4, iters=_log(rng, 50, 100))
    elif kind == "lm":
        case["iters"] = rng.randint(3, 15)
    elif kind == "mp":
        case.update(scales=rng.randint(1, 3), learned=rng.random() < 0.5, fresh=rng.random() < 0.3)
    elif kind == "keyframe":
        case.update(matched=max(200, n // rng.randint(10, 40)), per_gauss=rng.randint(1, 8))
    return case


# Contributions of Gaussians to a pixel in these scenes (a converged map's
# surfaces cover a pixel about 20 times over before it is opaque), and the
# operations of one: exponent, alpha and six channels forward; the same again
# with the chain to the parameters backward; six tangents for the Jacobian.
LAYERS, OPS_FWD, OPS_BWD, OPS_JAC = 20, 33, 70, 200


def work(case):
    k, P = case["kind"], case["width"] * case["height"]
    if k in ("infer", "train"):
        px = P * case["batch"]
        flops = px * 2 * (8 * 32 + 9 * 32 * 32 + 32 * 32 + 32)
        if k == "infer":
            return {"bytes": px * (16 + 4), "flops": flops}
        return {"bytes": px * (16 + 4) + 7 * 4 * dags.MPNET_PARAMS, "flops": 3 * flops}
    n = case["n"]
    V = case.get("views", 1)
    if k == "splat":
        image = 0 if case["autograd"] else P * (32 + 4)
        return {"bytes": n * 64 * 2 + P * 16 + image, "flops": P * LAYERS * (OPS_FWD + OPS_BWD)}
    if k == "render":
        return {"bytes": n * 64 * 2 + P * 4 * (6 + 4), "flops": P * LAYERS * (OPS_FWD + OPS_BWD)}
    if k == "mapping":
        # records, snapshot, moments, master colour; image, last and targets
        return {"bytes": n * (64 * 2 + 64 + 4 * 64 + 2 * 16 + 64) + V * P * (16 + 32 + 4),
                "flops": V * P * LAYERS * (OPS_FWD + OPS_BWD)}
    if k == "track":
        frames = case["frames"]
        return {"bytes": n * 64 + frames * P * (16 + 32 + 4),
                "flops": frames * case["iters"] * P * LAYERS * (OPS_FWD + OPS_BWD)}
    if k == "lm":
        return {"bytes": n * 64 + P * 16, "flops": case["iters"] * P * LAYERS * OPS_JAC}
    if k == "mp":
        flops = P * 60 + n * 13 * 12
        bytes_ = n * (64 + 4 + 1) + P * (16 + 16 + 1)
        if case["learned"]:
            flops += P * 2 * (8 * 32 + 9 * 32 * 32 + 32 * 32 + 32)
            bytes_ += P * (8 + 16 + 4)
        return {"bytes": bytes_, "flops": flops}
    m = case["matched"] * case["per_gauss"]
    return {"bytes": m * (8 + 8 + 4 + 4) + n * (4 + 1 + 4) + P * 4, "flops": m * 40}


# -------------------------------------------------------------------- scenes

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=F64)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=F64)


def _camera(case):
    w, h = case["width"], case["height"]
    f = 0.75 * w if case.get("scene") == "box" else 525.0 * w / 640
    return dags.Camera(f, f, w / 2.0, h / 2.0, w, h)


def _records(mean, logit, quat, logscale, mp, rgb):
    """The 64-byte records (float32 [n, 16]) of per-Gaussian tensors."""
    rec = torch.zeros((mean.shape[0], 16), dtype=torch.float32, device=DEV)
    rec[:, 0:3], rec[:, 3], rec[:, 4:8], rec[:, 8:11], rec[:, 11] = mean, logit, quat, logscale, mp
    rec.view(torch.bfloat16)[:, 24:27] = rgb.to(torch.float32)
    return rec


def _texture(p):
    return torch.stack([0.5 + 0.3 * torch.sin(2.1 * p[..., 0] + 0.7 * p[..., 2]) * torch.cos(1.3 * p[..., 1]),
                        0.5 + 0.3 * torch.sin(1.7 * p[..., 2] - 1.1 * p[..., 1] + 0.4),
                        0.5 + 0.3 * torch.cos(2.5 * p[..., 0] - 1.9 * p[..., 2] + 1.3 * p[..., 1])], -1)


def _box_map(n, g):
    """Anisotropic Gaussians in a box 1 to 4 m ahead, 20% of them a dynamic cluster."""
    lo = torch.tensor([-1.0, -1.0, 1.0], device=DEV, dtype=F64)
    mean = lo + _rand(g, n, 3) * torch.tensor([2.0, 2.0, 3.0], device=DEV, dtype=F64)
    nd = n // 5
    mean[:nd] = torch.tensor([0.2, -0.3, 1.5], device=DEV, dtype=F64) + \
        _rand(g, nd, 3) * torch.tensor([0.6, 0.6, 1.0], device=DEV, dtype=F64)
    quat = _randn(g, n, 4)
    quat = quat / quat.norm(dim=1, keepdim=True)
    mp = torch.full((n,), 0.1, device=DEV, dtype=F64)
    mp[:nd] = 0.9
    return _records(mean, _randn(g, n), quat, -3.0 + 0.5 * _randn(g, n, 3), mp, _rand(g, n, 3))


def _room_map(n, g):
    """Disc-like Gaussians covering the room's planes and the objects without
    holes, as in a converged map. Returns (records, object of each or -1)."""
    half, objs = synth.ROOM_HALF, synth.default_objects()
    areas, planes = [], [(0, -1), (0, 1), (2, -1), (2, 1), (1, -1), (1, 1)]
    for axis, _ in planes:
        a, b = [half[k] for k in range(3) if k != axis]
        areas.append(4 * a * b)
    for ob in objs:
        a, b, c = ob.axes ** 1.6
        areas.append(4 * math.pi * ((a * b + a * c + b * c) / 3) ** (1 / 1.6))
    areas = np.array(areas)
    counts = np.floor(n * areas / areas.sum()).astype(int)
    counts[0] += n - counts.sum()
    pts, normals, obj = [], [], []
    for (axis, sign), m in zip(planes, counts[:6]):
        o = [k for k in range(3) if k != axis]
        ex, ey = half[o[0]], half[o[1]]
        nx = max(1, int(math.sqrt(m * ex / ey)))
        ny = max(1, m // nx)
        k = torch.arange(m, device=DEV)
        cell = torch.stack([(k % (nx * ny)) // ny, (k % (nx * ny)) % ny], 1).to(F64) + 0.1 + 0.8 * _rand(g, m, 2)
        p = torch.full((m, 3), sign * half[axis], device=DEV, dtype=F64)
        p[:, o[0]], p[:, o[1]] = cell[:, 0] / nx * 2 * ex - ex, cell[:, 1] / ny * 2 * ey - ey
        nv = torch.zeros((m, 3), device=DEV, dtype=F64)
        nv[:, axis] = -sign
        pts.append(p), normals.append(nv), obj.append(torch.full((m,), -1, device=DEV))
    for j, (ob, m) in enumerate(zip(objs, counts[6:])):
        k = torch.arange(m, device=DEV, dtype=F64) + 0.5
        z, phi = 1 - 2 * k / max(1, m), math.pi * (1 + 5 ** 0.5) * k
        r = torch.sqrt(1 - z * z)
        d = torch.stack([r * torch.cos(phi), r * torch.sin(phi), z], 1)
        ax = torch.from_numpy(ob.axes).to(DEV)
        nv = d / ax
        pts.append(torch.from_numpy(ob.center).to(DEV) + d * ax)
        normals.append(nv / nv.norm(dim=1, keepdim=True)), obj.append(torch.full((int(m),), j, device=DEV))
    pts, nv, obj = torch.cat(pts), torch.cat(normals), torch.cat(obj)
    # the rotation that takes z to the normal
    quat = torch.stack([1 + nv[:, 2], -nv[:, 1], nv[:, 0], torch.zeros_like(nv[:, 0])], 1)
    quat[nv[:, 2] < -0.999999] = torch.tensor([0.0, 1.0, 0.0, 0.0], device=DEV, dtype=F64)
    quat = quat / quat.norm(dim=1, keepdim=True)
    ls = torch.full((n, 3), math.log(0.002), device=DEV, dtype=F64)
    ls[:, 0:2] = math.log(0.7 * math.sqrt(areas.sum() / n)) + 0.1 * _randn(g, n, 2)
    rgb = (_texture(pts) + 0.1 * (_rand(g, n, 3) - 0.5)).clamp(0, 1)
    moving = torch.zeros(n, dtype=torch.bool, device=DEV)
    for j, ob in enumerate(objs):
        if np.any(ob.velocity != 0):
            moving |= obj == j
    mp = torch.where(moving, 0.85, 0.1) + 0.1 * (_rand(g, n) - 0.5)
    return _records(pts, 4.0 + 0.5 * _randn(g, n), quat, ls, mp, rgb), obj, moving


def _raycast(cam, pose, t, g):
    """RGB-D of the room at time t from a world-to-camera pose (3x4 numpy):
    float64 [P, 4] with 1% depth noise (0 where the depth is outside 0.5-5 m),
    and the object each pixel sees (-1: the room)."""
    W, H = cam.width, cam.height
    jj, ii = torch.meshgrid(torch.arange(H, device=DEV, dtype=F64), torch.arange(W, device=DEV, dtype=F64),
                            indexing="ij")
    dc = torch.stack([(ii - cam.cx) / cam.fx, (jj - cam.cy) / cam.fy, torch.ones_like(ii)], -1).reshape(-1, 3)
    R = torch.from_numpy(np.ascontiguousarray(pose[:, :3])).to(DEV)
    dw = (dc[:, :, None] * R[None]).sum(1)
    ow = -(pose[:, :3].T @ pose[:, 3])
    best = torch.full((W * H,), math.inf, device=DEV, dtype=F64)
    hit = torch.full((W * H,), -1, device=DEV)
    for axis in range(3):
        for sign in (-1.0, 1.0):
            s = (sign * synth.ROOM_HALF[axis] - ow[axis]) / dw[:, axis]
            best = torch.where((s > 1e-6) & (s < best), s, best)
    for j, ob in enumerate(synth.default_objects()):
        oc = torch.from_numpy((ow - ob.center_at(t)) / ob.axes).to(DEV)
        dd = dw / torch.from_numpy(ob.axes).to(DEV)
        a, b, c = (dd * dd).sum(1), 2 * (dd * oc).sum(1), (oc * oc).sum() - 1
        disc = b * b - 4 * a * c
        s = (-b - torch.sqrt(disc.clamp(min=0))) / (2 * a)
        ok = (disc > 0) & (s > 1e-6) & (s < best)
        best, hit = torch.where(ok, s, best), torch.where(ok, torch.full_like(hit, j), hit)
    rgb = _texture(torch.from_numpy(ow).to(DEV) + best[:, None] * dw)
    depth = best * (1 + 0.01 * _randn(g, W * H))
    depth = torch.where((depth < 0.5) | (depth > 5.0), torch.zeros_like(depth), depth)
    return torch.cat([rgb, depth[:, None]], 1), hit


def _keyframe_poses(views, g):
    """Keyframes on a ring inside the room, looking inward."""
    out = []
    jitter = (0.1 * (_rand(g, views, 2) - 0.5)).cpu().numpy()
    for v in range(views):
        a = 2 * math.pi * v / views + jitter[v, 0]
        eye = np.array([1.6 * math.cos(a), -0.3 + jitter[v, 1], 1.6 * math.sin(a)])
        out.append(synth.look_at_pose(eye, np.array([-0.5 * math.cos(a), 0.4, -0.5 * math.sin(a)])))
    return out


def _frames(seed, gap):
    """The world-to-camera poses of a frame of the camera's path and of the one
    `gap` frames on, and their indexes."""
    f = 10 + seed % 40
    path = synth.camera_path(f + gap + 1, FPS)
    return path[f], path[f + gap], f, f + gap


def _gpu(pose):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(pose, np.float64).reshape(-1, 12))).to(DEV)


def _features(case, g):
    """Network input [B, H, W, 8] as frames give it (rendered MP, colour and
    depth residuals, depth, opacity, prior), smooth in space, and a target map."""
    B, H, W = case["batch"], case["height"], case["width"]
    coarse = torch.rand((B, 9, 1 + H // 16, 1 + W // 16), generator=g, device=DEV)
    x = torch.nn.functional.interpolate(coarse, size=(H, W), mode="bilinear", align_corners=False)
    noise = torch.rand((B, 5, H, W), generator=g, device=DEV)
    moving = (x[:, 0] > 0.7).float()
    feats = torch.empty((B, H, W, 8), dtype=torch.bfloat16, device=DEV)
    feats[..., 0] = 0.1 + 0.7 * moving * x[:, 1]
    for c in range(3):
        feats[..., 1 + c] = 0.05 * noise[:, c] + 0.3 * moving * x[:, 2 + c]
    feats[..., 4] = 0.02 * noise[:, 3] + 0.4 * moving * x[:, 5]
    feats[..., 5] = 0.5 + 4.5 * x[:, 6]
    feats[..., 6] = 1 - 0.05 * noise[:, 4]
    feats[..., 7] = torch.where(x[:, 0] > 0.72, 0.9, 0.1)
    target = (0.05 + 0.85 * moving * x[:, 1] + 0.05 * x[:, 7]).clamp(0, 1)
    target[x[:, 8] < 0.25] = -1.0            # pixels that the training leaves out
    return feats, target.contiguous()


def _inputs(case, seed):
    """The case's inputs, from the seed alone."""
    g, k = _gen(seed), case["kind"]
    s = {"case": case}
    if k in ("infer", "train"):
        blob, master = synth.mpnet_init(seed % 1000)
        s["weights"] = torch.from_numpy(blob).to(DEV)
        s["feats"], target = _features(case, g)
        if k == "train":
            n = dags.MPNET_PARAMS
            s.update(target=target, master=torch.from_numpy(master).to(DEV), step=200,
                     m=(2e-3 * _randn(g, n)).float(), v=(5e-3 * torch.exp(0.5 * _randn(g, n))).square().float())
        return s
    cam = s["cam"] = _camera(case)
    n, P = case["n"], cam.width * cam.height
    if case.get("scene") == "box":
        s["gauss"] = _box_map(n, g)
        s["poses"] = _gpu(synth.identity_pose())
        tg = torch.cat([_rand(g, P, 3), 1 + 3 * _rand(g, P, 1)], 1)
        s["targets"] = tg.float()[None]
        return s
    s["gauss"], obj, moving = _room_map(n, g)
    if k == "mapping":
        poses = _keyframe_poses(case["views"], g)
        s["poses"] = _gpu(np.stack(poses))
        s["targets"] = torch.stack([_raycast(cam, p, 0.0, g)[0].float() for p in poses])
        s["map"] = s["gauss"].clone()                       # the map at the start of the iteration
        s["prev"] = s["gauss"].clone()                      # the map after the previous one
        s["prev"][:, 0:3] += (0.002 * _randn(g, n, 3)).float()
        s["m"] = (0.3 * _randn(g, n, 16)).float()
        s["v"] = torch.exp(0.5 * _randn(g, n, 16)).float()
        s["colour"] = torch.zeros((n, 4), dtype=torch.float32, device=DEV)
        s["colour"][:, 0:3] = s["gauss"].view(torch.bfloat16)[:, 24:27].float()
        s["step"] = 100
        return s
    if k == "track":
        f0 = 10 + seed % 40
        path = synth.camera_path(f0 + case["frames"] + 1, FPS)
        s["poses"] = _gpu(np.stack(path[f0:f0 + case["frames"]]))
        s["frames"] = torch.stack([_raycast(cam, path[f0 + 1 + j], (f0 + 1 + j) / FPS, g)[0].float()
                                   for j in range(case["frames"])])
        return s
    before, now, f0, f1 = _frames(seed, 5 if k == "keyframe" else 1)
    tg, hit = _raycast(cam, now, f1 / FPS, g)
    s["targets"] = tg.float()[None]
    s["poses"] = _gpu(before)
    if k == "mp":
        # the render of the map at the tracked pose: the room as it was mapped
        # (the objects where they were), blended over a little of nothing
        img, seen = _raycast(cam, now, 0.0, g)
        o = 0.9 + 0.1 * _rand(g, P)
        mp = torch.where((seen >= 0) & (seen < 2), 0.85, 0.1) + 0.05 * _rand(g, P)
        d = torch.where(img[:, 3] > 0, img[:, 3], torch.full_like(o, 5.0))
        image = torch.cat([((img[:, 0:3] + 0.03 * _randn(g, P, 3)).clamp(0, 1) * o[:, None]).t(), (d * o)[None],
                           o[None], (o * mp)[None], (1 - o)[None], (1 - mp)[None]])
        s["image"] = image.float().contiguous()
        inst = torch.where((hit >= 0) & (hit < 2), hit + 1, torch.zeros_like(hit))
        flip = _rand(g, P) < 0.05
        s["inst"] = torch.where(flip, (inst + 1) % 3, inst).to(torch.uint8)
        s["table"] = torch.tensor([[0.1, 0.05], [0.9, 0.8], [0.85, 0.7]], dtype=torch.float32, device=DEV)
        s["labels"] = moving.to(torch.uint8)
        s["pose"] = _gpu(now)
        s["trigger"] = torch.zeros(2, dtype=torch.int32, device=DEV)
        if case["learned"]:
            s["weights"] = torch.from_numpy(synth.mpnet_init(seed % 1000)[0]).to(DEV)
        return s
    if k == "keyframe":
        other, _ = _raycast(cam, before, f0 / FPS, g)
        s["depth_i"], s["depth_j"] = other[:, 3].float().contiguous(), tg[:, 3].float().contiguous()
        s["weight_j"] = (1 - 0.9 * _rand(g, P) * (hit >= 0)).float()
        s["pose_i"], s["pose_j"] = _gpu(before), _gpu(now)
        vel = torch.zeros((n, 3), device=DEV, dtype=F64)
        for j, ob in enumerate(synth.default_objects()):
            vel[obj == j] = torch.from_numpy(ob.velocity).to(DEV)
        pix, ok = [], torch.ones(n, dtype=torch.bool, device=DEV)
        for pose, f in ((before, f0), (now, f1)):
            T = torch.from_numpy(pose).to(DEV)
            X = s["gauss"][:, 0:3].double() + vel * (f / FPS)
            Y = (X[:, None, :] * T[None, :, :3]).sum(2) + T[:, 3]
            u = torch.stack([cam.fx * Y[:, 0] / Y[:, 2] + cam.cx, cam.fy * Y[:, 1] / Y[:, 2] + cam.cy], 1)
            ok &= (Y[:, 2] > 0.3) & (u[:, 0] >= 0) & (u[:, 0] <= cam.width - 1) & (u[:, 1] >= 0) & \
                (u[:, 1] <= cam.height - 1)
            pix.append(u)
        cand = torch.nonzero(ok)[:, 0]
        pick = cand[torch.randperm(cand.shape[0], generator=g, device=DEV)[:case["matched"]]]
        gid = pick.repeat_interleave(case["per_gauss"])
        gid = gid[torch.randperm(gid.shape[0], generator=g, device=DEV)]
        s["gid"] = gid.int()
        s["p1"], s["p2"] = ((u[gid] + 0.3 * _randn(g, gid.shape[0], 2)).float().contiguous() for u in pix)
        labels = moving | (_rand(g, n) < 0.1)
        s["labels"] = labels.to(torch.uint8)
    return s


# ------------------------------------------------------------------- running

def prepare(case, seed):
    s = _inputs(case, seed)
    k = case["kind"]
    if k in ("infer", "train"):
        s["ctx"] = dags.Context(1024, case["width"], case["height"])
        s["out"] = torch.empty((case["batch"], case["height"], case["width"]), dtype=torch.float32, device=DEV)
        if k == "train":
            s["loss"] = torch.empty(1, dtype=F64, device=DEV)
            s["grad"] = torch.empty(dags.MPNET_PARAMS, dtype=torch.float32, device=DEV)
        return s
    cam, n = s["cam"], case["n"]
    V, P = case.get("views", 1), cam.width * cam.height
    s["ctx"] = dags.Context(n, cam.width, cam.height, V)
    buffers = k in ("mapping", "track") or not case.get("autograd", True)
    if k == "render":
        t = s["targets"][0].t().reshape(1, 4, cam.height, cam.width)
        s["rgb"], s["depth"] = t[:, 0:3].contiguous(), t[:, 3].contiguous()
    if k in ("splat", "render") and not buffers:
        s["gauss"].requires_grad_(True)
        s["xi"] = torch.zeros((1, 6), dtype=F64, device=DEV, requires_grad=True)
    if buffers:
        s["image"] = torch.empty((V, dags.IMG_CHANNELS, cam.height, cam.width), dtype=torch.float32, device=DEV)
        s["last"] = torch.empty((V, cam.height, cam.width), dtype=torch.int32, device=DEV)
        s["loss"] = torch.empty(1, dtype=F64, device=DEV)
    if buffers and k != "track":
        s["grad"] = torch.empty((n, dags.GRAD_WORDS), dtype=torch.float32, device=DEV)
        s["grad_pose"] = torch.empty((V, 6), dtype=F64, device=DEV)
    if k == "mapping":
        s["lmp"] = torch.empty(1, dtype=F64, device=DEV)
    if k in ("track", "lm"):
        s["pose"] = torch.empty(12, dtype=F64, device=DEV)
        s["cfg"] = dags.default_pose_cfg()
    if k == "track":
        s["target"] = torch.empty((1, P, 4), dtype=torch.float32, device=DEV)
        s["adam"] = torch.empty(13, dtype=F64, device=DEV)
        s["grad_pose"] = torch.empty(6, dtype=F64, device=DEV)
        s["tracked"] = torch.empty((case["frames"], 12), dtype=F64, device=DEV)
    if k == "lm":
        s["state"] = torch.empty(dags.LM_STATE, dtype=F64, device=DEV)
    if k == "mp":
        s["cfg"] = dags.default_mp_cfg(scales=case["scales"])
        s["stats"] = torch.empty(dags.MP_STATS_HEAD + 4 * 3, dtype=F64, device=DEV)
        if case["learned"]:
            s["feats"] = torch.empty((1, cam.height, cam.width, 8), dtype=torch.bfloat16, device=DEV)
            s["mp_map"] = torch.empty((1, cam.height, cam.width), dtype=torch.float32, device=DEV)
    if k == "keyframe":
        s["edge"] = torch.empty(13, dtype=F64, device=DEV)
    return s


def _own_loss(C, D, O, R, rgb, depth):
    """A caller's own loss on rendered channels: squared colour, absolute depth,
    and a pull of the opacity to one away from moving objects."""
    f = torch.nn.functional
    return f.mse_loss(C, rgb, reduction="sum") + 0.1 * f.l1_loss(D, depth, reduction="sum") + \
        0.01 * ((1 - O) * (1 - R)).sum()


def run(s):
    case, ctx = s["case"], s["ctx"]
    k = case["kind"]
    if k == "infer":
        return {"mp": ctx.mpnet_infer(s["weights"], s["feats"], out=s["out"])}
    if k == "train":
        s["step"] += 1
        loss = ctx.mpnet_train_step(s["weights"], s["master"], s["m"], s["v"], s["step"], s["feats"], s["target"],
                                    1e-3, loss=s["loss"], grad=s["grad"])
        return {"loss": loss, "grad": s["grad"], "master": s["master"], "m": s["m"], "v": s["v"],
                "w": s["weights"][:21568].view(torch.bfloat16), "b": s["weights"][21568:21956].view(torch.float32)}
    cam, gauss = s["cam"], s["gauss"]
    if k == "splat" and not case["autograd"]:
        ctx.forward(gauss, cam, s["poses"], s["targets"], image=s["image"], last=s["last"], loss=s["loss"])
        ctx.backward(gauss, cam, s["poses"], s["targets"], s["image"], s["last"], dags.GRAD_GAUSS | dags.GRAD_POSE,
                     grad_gauss=s["grad"], grad_pose=s["grad_pose"])
        return {"image": s["image"], "last": s["last"], "loss": s["loss"], "gauss": s["grad"], "xi": s["grad_pose"]}
    if k == "splat":
        gauss.grad = s["xi"].grad = None
        loss = autograd.splat_loss(ctx, cam, gauss, s["poses"], s["targets"], s["xi"])
        loss.sum().backward()
        return {"loss": loss.detach(), "gauss": gauss.grad, "xi": s["xi"].grad}
    if k == "render":
        gauss.grad = s["xi"].grad = None
        C, D, O, R = autograd.splat_render(ctx, cam, gauss, s["poses"], s["xi"])
        loss = _own_loss(C, D, O, R, s["rgb"], s["depth"])
        loss.backward()
        return {"C": C.detach(), "D": D.detach(), "O": O.detach(), "R": R.detach(), "loss": loss.detach(),
                "gauss": gauss.grad, "xi": s["xi"].grad}
    if k == "mapping":
        gauss.copy_(s["map"])      # every pass is the same iteration of the window
        ctx.forward(gauss, cam, s["poses"], s["targets"], image=s["image"], last=s["last"], loss=s["loss"])
        ctx.backward(gauss, cam, s["poses"], s["targets"], s["image"], s["last"], dags.GRAD_GAUSS,
                     grad_gauss=s["grad"])
        ctx.mp_consistency(gauss, s["prev"], grad=s["grad"], loss=s["lmp"])
        ctx.gauss_adam_step(gauss, (s["colour"], s["m"], s["v"]), s["grad"], s["step"])
        return {"image": s["image"], "last": s["last"], "loss": s["loss"], "lmp": s["lmp"], "grad": s["grad"],
                "params": gauss[:, 0:12], "rgb": gauss.view(torch.bfloat16)[:, 24:27], "colour": s["colour"],
                "m": s["m"], "v": s["v"]}
    if k == "track":
        for j in range(case["frames"]):
            s["target"].copy_(s["frames"][j:j + 1])
            s["pose"].copy_(s["poses"][j])
            s["adam"].zero_()
            ctx.track(gauss, cam, s["pose"], s["target"], case["iters"], s["adam"], s["image"], s["last"], s["loss"],
                      s["grad_pose"], pcfg=s["cfg"])
            s["tracked"][j].copy_(s["pose"])
        return {"poses": s["tracked"]}
    if k == "lm":
        s["pose"].copy_(s["poses"][0])
        ctx.track_lm(gauss, cam, s["pose"], s["targets"][0], case["iters"], state=s["state"])
        return {"pose": s["pose"], "state": s["state"]}
    if k == "mp":
        mp_map = None
        out = {}
        if case["learned"]:
            ctx.mpnet_features(s["image"], s["targets"][0], s["inst"], s["table"], cam, out=s["feats"][0])
            mp_map = ctx.mpnet_infer(s["weights"], s["feats"], out=s["mp_map"])
            out = {"feats": s["feats"], "mp_map": mp_map}
        ctx.mp_update(gauss, cam, s["pose"], s["targets"][0], s["image"], s["inst"], s["table"], s["labels"],
                      cfg=s["cfg"], seg_refreshed=case["fresh"], stats=s["stats"], mp_map=mp_map)
        ctx.semantic_trigger(s["stats"], s["trigger"], case["fresh"])
        return {**out, "gauss": gauss, "labels": s["labels"], "stats": s["stats"], "trigger": s["trigger"]}
    d, dbar = ctx.epipolar_verify(cam, s["pose_i"], s["pose_j"], s["p1"], s["p2"], s["gid"], gauss, s["labels"])
    edge = ctx.edge_warp(cam, s["depth_i"], s["depth_j"], s["weight_j"], s["pose_i"], s["pose_j"], out=s["edge"])
    return {"d": d, "dbar": dbar, "gauss": gauss, "labels": s["labels"], "edge": edge}


# --------------------------------------------------------- the same, in 64 bits

def _fields(rec):
    """The optimised parameters of records, as float64 tensors."""
    r = rec.double()
    return [r[:, 0:3].clone(), r[:, 3].clone(), r[:, 4:8].clone(), r[:, 8:11].clone(),
            rec.view(torch.bfloat16)[:, 24:27].double()]


def _project(fields, mp, pose, xi, cam):
    """Projected Gaussians (u, v, conic a b c, opacity, depth, r, g, b, MP as the
    rows of one matrix) and the 2D variances, at exp(xi^) pose to first order."""
    mean, logit, quat, ls, rgb = fields
    rho, phi = xi[0:3], xi[3:6]
    zero = torch.zeros_like(phi[0])
    hat = torch.stack([torch.stack([zero, -phi[2], phi[1]]), torch.stack([phi[2], zero, -phi[0]]),
                       torch.stack([-phi[1], phi[0], zero])])
    R0, t0 = pose[:, :3], pose[:, 3]
    R, t = R0 + hat @ R0, t0 + hat @ t0 + rho
    p = mean @ R.t() + t
    x, y, z = p.unbind(1)
    q = quat / quat.norm(dim=1, keepdim=True)
    w, a, b, c = q.unbind(1)
    Rq = torch.stack([1 - 2 * (b * b + c * c), 2 * (a * b - w * c), 2 * (a * c + w * b),
                      2 * (a * b + w * c), 1 - 2 * (a * a + c * c), 2 * (b * c - w * a),
                      2 * (a * c - w * b), 2 * (b * c + w * a), 1 - 2 * (a * a + b * b)], 1).reshape(-1, 3, 3)
    K = torch.einsum("ij,njk->nik", R, Rq) * torch.exp(ls)[:, None, :]
    lx, ly = GUARD * 0.5 * cam.width / cam.fx, GUARD * 0.5 * cam.height / cam.fy
    tx, ty = (x / z).clamp(-lx, lx), (y / z).clamp(-ly, ly)
    m0 = (cam.fx / z)[:, None] * K[:, 0] - (cam.fx * tx / z)[:, None] * K[:, 2]
    m1 = (cam.fy / z)[:, None] * K[:, 1] - (cam.fy * ty / z)[:, None] * K[:, 2]
    A, B, C = (m0 * m0).sum(1) + DILATION, (m0 * m1).sum(1), (m1 * m1).sum(1) + DILATION
    det = A * C - B * B
    o = torch.sigmoid(logit)
    rows = torch.stack([cam.fx * x / z + cam.cx, cam.fy * y / z + cam.cy, C / det, -B / det, A / det, o, z,
                        rgb[:, 0], rgb[:, 1], rgb[:, 2], mp], 1)
    return rows, A, C


def _tiles(rec, pose, cam):
    """The Gaussians that reach the image, and each tile's list of them in depth
    order: (ids, list [pairs], start [tiles + 1]). The order is that of the FP32
    camera depth, ties by id, as the library defines it."""
    with torch.no_grad():
        fields = _fields(rec)
        rows, A, C = _project(fields, rec[:, 11].double(), pose, torch.zeros(6, device=DEV, dtype=F64), cam)
        u, v, o, z = rows[:, 0], rows[:, 1], rows[:, 5], rows[:, 6]
        p32 = pose.float()
        d32 = ((p32[2, 0] * rec[:, 0] + p32[2, 1] * rec[:, 1]) + p32[2, 2] * rec[:, 2]) + p32[2, 3]
        grow = torch.sqrt(2 * torch.log((o / ALPHA_MIN).clamp(min=1)))
        ex, ey = grow * torch.sqrt(A) + 1e-3, grow * torch.sqrt(C) + 1e-3
        tw, th = -(-cam.width // TILE), -(-cam.height // TILE)
        ok = (z > Z_NEAR) & (o > ALPHA_MIN) & torch.isfinite(u) & torch.isfinite(v)

        def cell(t, most):
            return torch.where(ok, t, torch.zeros_like(t)).div(TILE).floor().clamp(0, most).long()

        x0, x1 = cell(u - ex, tw), torch.where(ok, cell(u + ex + TILE, tw), torch.zeros_like(d32, dtype=torch.long))
        y0, y1 = cell(v - ey, th), cell(v + ey + TILE, th)
        count = ((x1 - x0).clamp(min=0) * (y1 - y0).clamp(min=0))
        ids = torch.nonzero(count)[:, 0]
        ids = ids[torch.sort(d32[ids], stable=True).indices]       # depth order, ties by id
        x0, y0, cw, m = x0[ids], y0[ids], (x1 - x0)[ids], count[ids]
        rank = torch.arange(ids.shape[0], device=DEV).repeat_interleave(m)
        j = torch.arange(rank.shape[0], device=DEV) - (torch.cumsum(m, 0) - m)[rank]
        tile = (y0[rank] + j // cw[rank]) * tw + x0[rank] + j % cw[rank]
        order = torch.sort(tile, stable=True)
        start = torch.searchsorted(order.values, torch.arange(tw * th + 1, device=DEV))
        return ids, rank[order.indices], start


def _composite(rows, lst, tiles, start, cam):
    """Front-to-back compositing of some tiles: channels [tiles, 256, 6] (r, g,
    b, depth, opacity, MP), final transmittance, pixel index, inside the image."""
    s, e = start[tiles], start[tiles + 1]
    L = max(1, int((e - s).max()))
    k = s[:, None] + torch.arange(L, device=DEV)
    valid = k < e[:, None]
    f = rows[lst[k.clamp(max=max(0, lst.shape[0] - 1))]] if lst.shape[0] else rows.new_zeros((*k.shape, 11))
    tw = -(-cam.width // TILE)
    px = (tiles % tw)[:, None] * TILE + torch.arange(256, device=DEV) % TILE
    py = (tiles // tw)[:, None] * TILE + torch.arange(256, device=DEV) // TILE
    f = f[:, :, None, :]
    dx, dy = f[..., 0] - px[:, None, :], f[..., 1] - py[:, None, :]
    ag = f[..., 5] * torch.exp(-0.5 * (f[..., 2] * dx * dx + 2 * f[..., 3] * dx * dy + f[..., 4] * dy * dy))
    live = valid[:, :, None] & (ag >= ALPHA_MIN)
    alpha = torch.where(live, ag.clamp(max=ALPHA_MAX), torch.zeros_like(ag))
    with torch.no_grad():
        keep = torch.cumsum(torch.log1p(-alpha), 1) >= math.log(T_MIN)
    lt = torch.log1p(-torch.where(keep, alpha, torch.zeros_like(alpha)))
    cum = torch.cumsum(lt, 1)
    w = torch.where(keep, alpha, torch.zeros_like(alpha)) * torch.exp(cum - lt)
    chan = torch.stack([(w * f[..., c]).sum(1) for c in (7, 8, 9, 6)] + [w.sum(1), (w * f[..., 10]).sum(1)], -1)
    return chan, torch.exp(cum[:, -1]), py * cam.width + px, (px < cam.width) & (py < cam.height)


def _chunks(start, budget=1 << 25):
    """Tiles in groups of like list lengths, so that a group's padded lists hold
    about `budget` pixel-Gaussian pairs."""
    length = start[1:] - start[:-1]
    order = torch.sort(length, descending=True)
    lens, at = order.values.tolist(), 0
    while at < len(lens):
        c = max(1, budget // (256 * max(1, lens[at])))
        yield order.indices[at:at + c]
        at += c


def _loss_terms(chan, tg, inside):
    """The MP-weighted loss of pixels (weights constant in the adjoint)."""
    o, rm = chan[..., 4], chan[..., 5]
    wgt = torch.where(o > 1e-6, (o - rm) / o.clamp(min=1e-300), torch.zeros_like(o)).detach()
    l1 = (chan[..., 0:3] - tg[..., 0:3]).abs().sum(-1)
    ld = torch.where(tg[..., 3] > 0, (chan[..., 3] - tg[..., 3]).abs(), torch.zeros_like(o))
    return torch.where(inside, wgt * (0.9 * l1 + 0.1 * ld), torch.zeros_like(o)), wgt


def _view(rec, fields, pose, xi, cam, targets, own=None):
    """Image [8, P] and loss of one view; gradients are added to the leaves
    `fields` and `xi`. own: the caller's gradient of channels, from the image."""
    P = cam.width * cam.height
    ids, lst, start = _tiles(rec, pose, cam)
    image = torch.zeros((8, P), device=DEV, dtype=F64)
    rows, _, _ = _project([t[ids] for t in fields], rec[ids, 11].double(), pose, xi, cam)
    leaf = rows.detach().requires_grad_(True)
    loss = torch.zeros((), device=DEV, dtype=F64)
    up = None
    for final in ((False, True) if own else (True,)):
        for tiles in _chunks(start):
            chan, T, pix, inside = _composite(leaf, lst, tiles, start, cam)
            pixc = torch.where(inside, pix, torch.zeros_like(pix))
            terms, wgt = _loss_terms(chan, targets[pixc].double(), inside)
            at = pix[inside]
            with torch.no_grad():
                image[0:6, at], image[6, at], image[7, at] = chan[inside].t(), T[inside], wgt[inside]
            if not final:
                continue
            if own:
                (chan * up[:, pixc].permute(1, 2, 0) * inside[..., None]).sum().backward()
            else:
                terms.sum().backward()
                loss += terms.detach().sum()
        if own and not final:
            up, loss = own(image)
    if leaf.grad is not None:
        rows.backward(leaf.grad)
    return image, loss


def _splat_grads(s, own=None):
    """Images, loss, record gradients [n, 16] and twist gradients [V, 6]."""
    rec, cam = s["gauss"].detach(), s["cam"]
    fields = [t.requires_grad_(True) for t in _fields(rec)]
    images, loss, gx = [], 0.0, []
    for v in range(s["poses"].shape[0]):
        xi = torch.zeros(6, device=DEV, dtype=F64, requires_grad=True)
        image, one = _view(rec, fields, s["poses"][v].reshape(3, 4), xi, cam, s["targets"][v], own)
        images.append(image.reshape(8, cam.height, cam.width))
        loss = loss + one
        gx.append(xi.grad if xi.grad is not None else torch.zeros_like(xi))
    grad = torch.zeros((rec.shape[0], 16), device=DEV, dtype=F64)
    for sl, t in zip((slice(0, 3), 3, slice(4, 8), slice(8, 11), slice(12, 15)), fields):
        if t.grad is not None:
            grad[:, sl] = t.grad
    return torch.stack(images), loss.reshape(1), grad, torch.stack(gx)


def _exact_splat(s):
    image, loss, grad, gx = _splat_grads(s)
    out = {"loss": loss, "gauss": grad, "xi": gx}
    return out if s["case"]["autograd"] else {**out, "image": image, "last": None}


def _exact_render(s):
    cam = s["cam"]

    def own(image):
        c = image[0:6].reshape(1, 6, cam.height, cam.width).clone().requires_grad_(True)
        tg = s["targets"].double().reshape(1, cam.height, cam.width, 4)
        loss = _own_loss(c[:, 0:3], c[:, 3], c[:, 4], c[:, 5], tg[..., 0:3].permute(0, 3, 1, 2), tg[..., 3])
        loss.backward()
        return c.grad.reshape(6, -1), loss.detach()

    image, loss, grad, gx = _splat_grads(s, own)
    return {"C": image[:, 0:3], "D": image[:, 3], "O": image[:, 4], "R": image[:, 5], "loss": loss.reshape(()),
            "gauss": grad, "xi": gx}


def _exact_mapping(s):
    image, loss, grad, _ = _splat_grads(s)
    rec, m, v = s["gauss"].double(), s["m"].double(), s["v"].double()
    mbar = (1 - rec[:, 11])[:, None]
    d = rec[:, 0:3] - s["prev"][:, 0:3].double()
    lmp = 500.0 * (mbar * d * d).sum().reshape(1)
    grad[:, 0:3] += 1000.0 * mbar * d
    lr = torch.tensor([1e-3] * 3 + [0.05] + [1e-3] * 4 + [5e-3] * 3 + [0.0] + [2.5e-3] * 3 + [0.0], device=DEV, dtype=F64)
    used = lr > 0
    m2 = torch.where(used, 0.9 * m + 0.1 * grad, m)
    v2 = torch.where(used, 0.999 * v + 0.001 * grad * grad, v)
    step = lr * (m2 / (1 - 0.9 ** s["step"])) / (torch.sqrt(v2 / (1 - 0.999 ** s["step"])) + 1e-8)
    colour = s["colour"].double()
    colour[:, 0:3] -= step[:, 12:15]
    return {"image": image, "last": None, "loss": loss, "lmp": lmp, "grad": grad, "params": (rec - step)[:, 0:12],
            "rgb": colour[:, 0:3], "colour": colour, "m": m2, "v": v2}


def _exp_se3(xi):
    """The rigid motion exp(xi^) (translation part first) as a 4x4 matrix."""
    M = torch.zeros((4, 4), device=DEV, dtype=F64)
    M[0, 1], M[0, 2], M[1, 2] = -xi[5], xi[4], -xi[3]
    M[1, 0], M[2, 0], M[2, 1] = xi[5], -xi[4], xi[3]
    M[0:3, 3] = xi[0:3]
    return torch.linalg.matrix_exp(M)


def _normal_equations(rec, pose, cam, targets):
    """(L, H, g) of the reweighted MP-weighted L1 loss at a pose, by forward-mode
    differentiation along the six twist directions."""
    ad = torch.autograd.forward_ad
    ids, lst, start = _tiles(rec, pose, cam)
    fields = [t[ids] for t in _fields(rec)]
    mp = rec[ids, 11].double()
    L = torch.zeros((), device=DEV, dtype=F64)
    H, g = torch.zeros((6, 6), device=DEV, dtype=F64), torch.zeros(6, device=DEV, dtype=F64)
    for tiles in _chunks(start):
        J = []
        for k in range(6):
            with torch.no_grad(), ad.dual_level():
                e = torch.zeros(6, device=DEV, dtype=F64)
                e[k] = 1.0
                xi = ad.make_dual(torch.zeros(6, device=DEV, dtype=F64), e)
                rows, _, _ = _project(fields, mp, pose, xi, cam)
                chan, _, pix, inside = _composite(rows, lst, tiles, start, cam)
                chan, tangent = ad.unpack_dual(chan)
                J.append(tangent[..., 0:4])
        J = torch.stack(J, -1)                              # [tiles, 256, 4, 6]
        tg = targets[torch.where(inside, pix, torch.zeros_like(pix))].double()
        terms, wgt = _loss_terms(chan, tg, inside)
        coef = wgt[..., None] * torch.tensor([0.9, 0.9, 0.9, 0.1], device=DEV, dtype=F64) * inside[..., None]
        coef[..., 3] *= tg[..., 3] > 0
        r = chan[..., 0:4] - tg
        W = coef / r.abs().clamp(min=0.01)
        L += terms.sum()
        H += torch.einsum("tpca,tpc,tpcb->ab", J, W, J)
        g += torch.einsum("tpca,tpc->a", J, W * r)
    return L, H, g


def _exact_lm(s):
    """Damped Gauss-Newton steps with accept and reject, from the starting pose."""
    rec, cam, tg = s["gauss"], s["cam"], s["targets"][0]
    best = tried = s["poses"][0].reshape(3, 4)
    L, mu, taken, H, g, last, ok = math.inf, 1e-2, 0, None, None, 0.0, False
    iu = torch.triu_indices(6, 6, device=DEV)
    for _ in range(s["case"]["iters"]):
        l1, h1, g1 = _normal_equations(rec, tried, cam, tg)
        last, ok = float(l1), float(l1) < L
        if ok:
            best, L, H, g, mu, taken = tried, last, h1, g1, max(mu * 0.1, 1e-9), taken + 1
        else:
            mu = min(mu * 10.0, 1e9)
        A = H + torch.diag(mu * torch.diagonal(H) + 1e-9 * torch.trace(H) / 6)
        E = _exp_se3(torch.linalg.solve(A, -g))
        tried = E[0:3, 0:3] @ best
        tried = torch.cat([tried[:, 0:3], tried[:, 3:4] + E[0:3, 3:4]], 1)
    state = torch.zeros(dags.LM_STATE, device=DEV, dtype=F64)
    state[0:12], state[12], state[13], state[14:35], state[35:41] = best.reshape(12), L, mu, H[iu[0], iu[1]], g
    state[41], state[42], state[43], state[44] = taken, s["case"]["iters"], last, float(ok)
    return {"pose": best.reshape(12), "state": state}


def _bf16(x):
    """x as BF16 holds it (its derivative that of x)."""
    return x + (x.detach().float().bfloat16().double() - x.detach())


def _net(weights, feats):
    """The network on one image: features [H, W, 8] and weights (W1, W2, W3, w4,
    b1, b2, b3, b4) in 64 bits; activations are held in BF16. Returns the logits."""
    W1, W2, W3, w4, b1, b2, b3, b4 = weights
    H, W, _ = feats.shape
    a1 = _bf16(torch.relu(feats.reshape(-1, 8) @ W1[:, :8].t() + b1)).reshape(H, W, 32)
    a1 = torch.nn.functional.pad(a1, (0, 0, 1, 1, 1, 1))
    z2 = b2
    for ky in range(3):
        for kx in range(3):
            c = (ky * 3 + kx) * 32
            z2 = z2 + a1[ky:ky + H, kx:kx + W].reshape(-1, 32) @ W2[:, c:c + 32].t()
    a3 = _bf16(torch.relu(_bf16(torch.relu(z2)) @ W3.t() + b3))
    return (a3 @ w4 + b4).reshape(H, W)


def _net_weights(blob):
    w, b = blob[:21568].view(torch.bfloat16).double(), blob[21568:21956].view(torch.float32).double()
    return [w[:512].reshape(32, 16), w[512:9728].reshape(32, 288), w[9728:10752].reshape(32, 32), w[10752:10784],
            b[0:32], b[32:64], b[64:96], b[96]]


def _exact_infer(s):
    w = _net_weights(s["weights"])
    return {"mp": torch.stack([torch.sigmoid(_net(w, f.double())) for f in s["feats"]])}


def _exact_train(s):
    w = [t.clone().requires_grad_(True) for t in _net_weights(s["weights"])]
    valid = s["target"] >= 0
    count = valid.sum().clamp(min=1)
    loss = 0.0
    for f, t, ok in zip(s["feats"], s["target"].double(), valid):
        z = _net(w, f.double())
        one = torch.where(ok, torch.nn.functional.softplus(z) - t * z, torch.zeros_like(z)).sum() / count
        one.backward()
        loss = loss + one.detach()
    grad = torch.cat([t.grad.reshape(-1) for t in w])
    step = s["step"] + 1
    m = 0.9 * s["m"].double() + 0.1 * grad
    v = 0.999 * s["v"].double() + 0.001 * grad * grad
    master = s["master"].double() - 1e-3 * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    pad = (torch.arange(512, device=DEV) % 16) >= 8         # the padded input channels stay zero
    master[:512][pad] = 0.0
    return {"loss": loss.reshape(1), "grad": grad, "master": master, "m": m, "v": v, "w": master[:10784],
            "b": master[10784:]}


def _disk_std(e, W, H):
    """Population standard deviation of a map over each pixel's disk of radius 2."""
    pad = torch.nn.functional.pad(e.reshape(1, 1, H, W), (2, 2, 2, 2), value=math.nan)[0, 0]
    win = torch.stack([pad[2 + j:2 + j + H, 2 + i:2 + i + W] for j in range(-2, 3) for i in range(-2, 3)
                       if i * i + j * j <= 4])
    inside = ~torch.isnan(win)
    n = inside.sum(0)
    mean = torch.where(inside, win, torch.zeros_like(win)).sum(0) / n
    return torch.sqrt(torch.where(inside, (win - mean) ** 2, torch.zeros_like(win)).sum(0) / n).reshape(-1)


def _lower_median(x):
    return torch.sort(x).values[(x.shape[0] - 1) // 2]


def _exact_mp(s):
    case, cam = s["case"], s["cam"]
    W, H = cam.width, cam.height
    img, tg, tab = s["image"].double(), s["targets"][0].double(), s["table"].double()
    inst = s["inst"].long()
    out = {}
    res = torch.where(tg[:, 3] > 0, (tg[:, 3] - img[3]).abs(), torch.zeros_like(img[3]))
    if case["learned"]:
        feats = torch.stack([img[5], *(tg[:, c] - img[c] for c in range(3)), res,
                             torch.where(tg[:, 3] > 0, tg[:, 3], torch.zeros_like(res)), img[4], tab[inst, 0]], -1)
        feats[:, 1:4] = feats[:, 1:4].abs()
        feats = feats.float().bfloat16().double().reshape(H, W, 8)
        external = torch.sigmoid(_net(_net_weights(s["weights"]), feats))
        out = {"feats": feats[None], "mp_map": external[None]}
    e = res + 0.05 * (tg[:, 0:3] - img[0:3].t()).abs().sum(1)
    nreg = tab.shape[0]
    cnt = torch.zeros(nreg, device=DEV, dtype=F64).index_add_(0, inst, torch.ones_like(e))
    mean = torch.zeros(nreg, device=DEV, dtype=F64).index_add_(0, inst, e) / cnt.clamp(min=1)
    var = torch.zeros(nreg, device=DEV, dtype=F64).index_add_(0, inst, (e - mean[inst]) ** 2) / cnt.clamp(min=1)
    sd = torch.sqrt(var)
    eub = (mean + 2.0 * sd).clamp(min=0.05)
    geo = torch.where(inst == 0, torch.exp(-_disk_std(e, W, H) / 0.05), torch.exp(-sd / 0.05)[inst])
    flat = (inst >= 1) & (sd < 0.005)[inst]
    m_geo = (torch.where(flat, mean[inst], e) / eub[inst]).clamp(0, 1)
    K = geo / (tab[inst, 1] + geo)
    mpix = (1 - K) * tab[inst, 0] + K * m_geo
    level = (external.reshape(H, W) if case["learned"] else mpix.reshape(H, W), e.reshape(H, W), img[3].reshape(H, W))
    rec = s["gauss"].double()
    T = s["pose"].reshape(3, 4)
    X = rec[:, 0:3] @ T[:, :3].t() + T[:, 3]
    z = X[:, 2]
    u, v = cam.fx * X[:, 0] / z + cam.cx, cam.fy * X[:, 1] / z + cam.cy
    n = rec.shape[0]
    vals, wts, oks, dmax = [[], []], [], [], torch.full((n,), -math.inf, device=DEV, dtype=F64)
    for sc in range(case["scales"]):
        if sc:
            def box(t, fn):
                h, w = t.shape[0] // 2, t.shape[1] // 2
                return fn(t[:2 * h, :2 * w].reshape(h, 2, w, 2))
            level = (box(level[0], lambda t: t.mean((1, 3))), box(level[1], lambda t: t.mean((1, 3))),
                     box(level[2], lambda t: t.amax((1, 3))))
        hs, ws = level[0].shape
        us, vs = u / 2 ** sc, v / 2 ** sc
        i0, j0 = torch.ceil(us - 2), torch.ceil(vs - 2)
        for dj in range(5):
            for di in range(5):
                i, j = i0 + di, j0 + dj
                d2 = (i - us) ** 2 + (j - vs) ** 2
                ok = (z > 0.2) & (d2 <= 4) & (i >= 0) & (i < ws) & (j >= 0) & (j < hs)
                p = torch.where(ok, j * ws + i, torch.zeros_like(i)).long()
                vals[0].append(level[0].reshape(-1)[p]), vals[1].append(level[1].reshape(-1)[p])
                wts.append(torch.where(ok, 2.0 ** -sc * torch.exp(-d2 / 2), torch.zeros_like(d2))), oks.append(ok)
                dmax = torch.where(ok, torch.maximum(dmax, level[2].reshape(-1)[p]), dmax)
    ok, wt = torch.stack(oks), torch.stack(wts)
    mv, ev = torch.stack(vals[0]), torch.stack(vals[1])
    c = ok.sum(0)
    seen = (c > 0) & ~((dmax > 0) & (z > dmax + 0.1))
    c1 = c.clamp(min=1)
    m_hat = (wt * mv).sum(0) / torch.where(seen, wt.sum(0), torch.ones_like(z))

    def variance(t):
        mu = torch.where(ok, t, torch.zeros_like(t)).sum(0) / c1
        return torch.where(ok, (t - mu) ** 2, torch.zeros_like(t)).sum(0) / c1

    M0 = rec[:, 11]
    U = -M0 * torch.log(M0 + 1e-6) - (1 - M0) * torch.log(1 - M0 + 1e-6) + variance(mv)
    u_min, u_max = U[seen].min(), U[seen].max()
    ut = (U - u_min) / (u_max - u_min)
    a = (0.05 + 0.55 * (1 - ut) * torch.exp(-torch.sqrt(variance(ev)) / 0.05)).clamp(0.05, 0.6)
    if not case["fresh"]:
        a = a * 0.5
    Mt = torch.where(seen, (1 - a) * M0 + a * m_hat, M0)
    rec[:, 11] = Mt
    med, u_bar = _lower_median(Mt[seen]), _lower_median(ut[seen])
    regions = torch.stack([cnt, mean, sd, eub], 1).reshape(-1)
    stats = torch.cat([torch.stack([med.clamp(min=0.5), u_bar, med, u_min, u_max, seen.sum().double()]), regions])
    return {**out, "gauss": rec, "labels": None, "stats": stats, "trigger": None}


def _exact_keyframe(s):
    cam = s["cam"]
    Ti, Tj = s["pose_i"].reshape(3, 4), s["pose_j"].reshape(3, 4)
    R = Tj[:, :3] @ Ti[:, :3].t()
    t = Tj[:, 3] - R @ Ti[:, 3]
    zero = torch.zeros((), device=DEV, dtype=F64)
    tx = torch.stack([torch.stack([zero, -t[2], t[1]]), torch.stack([t[2], zero, -t[0]]),
                      torch.stack([-t[1], t[0], zero])])
    Ki = torch.tensor([[1 / cam.fx, 0, -cam.cx / cam.fx], [0, 1 / cam.fy, -cam.cy / cam.fy], [0, 0, 1]], device=DEV,
                      dtype=F64)
    F = Ki.t() @ tx @ R @ Ki
    one = torch.ones((s["gid"].shape[0], 1), device=DEV, dtype=F64)
    line = torch.cat([s["p1"].double(), one], 1) @ F.t()
    den = torch.sqrt(line[:, 0] ** 2 + line[:, 1] ** 2)
    d = (torch.cat([s["p2"].double(), one], 1) * line).sum(1).abs() / den
    # lower median of each Gaussian's matches
    n, gid = s["case"]["n"], s["gid"].long()
    by_d = torch.sort(d)
    by_g = torch.sort(gid[by_d.indices], stable=True)
    sorted_d = by_d.values[by_g.indices]
    count = torch.bincount(gid, minlength=n)
    first = torch.cumsum(count, 0) - count
    at = (first + (count - 1).clamp(min=0) // 2).clamp(max=max(0, d.shape[0] - 1))
    dbar = torch.where(count > 0, sorted_d[at], torch.full((n,), math.nan, device=DEV, dtype=F64))
    rec = s["gauss"].double()
    back = (count > 0) & (dbar < 1.0) & (s["labels"] == 1)
    rec[:, 11] = torch.where(back, rec[:, 11].clamp(max=float(np.float32(0.1))), rec[:, 11])
    return {"d": d, "dbar": dbar, "gauss": rec, "labels": None, "edge": _edge(s, Ti, Tj)}


def _edge(s, Ti, Tj):
    """lambda L_edge and its gradients along both poses' twists."""
    cam = s["cam"]
    W, H = cam.width, cam.height
    Di, Dj, w = (s[k].double().reshape(H, W) for k in ("depth_i", "depth_j", "weight_j"))
    edge = torch.zeros((H, W), dtype=torch.bool, device=DEV)
    for dim in (0, 1):
        a, b = Di.narrow(dim, 0, Di.shape[dim] - 1), Di.narrow(dim, 1, Di.shape[dim] - 1)
        both, jump = (a > 0) & (b > 0), (a - b).abs()
        edge.narrow(dim, 0, Di.shape[dim] - 1).logical_or_(both & (jump > 0.05 * a))
        edge.narrow(dim, 1, Di.shape[dim] - 1).logical_or_(both & (jump > 0.05 * b))
    y, x = torch.nonzero(edge, as_tuple=True)
    d = Di[y, x]
    X = torch.stack([d * (x - cam.cx) / cam.fx, d * (y - cam.cy) / cam.fy, d], 1)
    xi_i, xi_j = (torch.zeros(6, device=DEV, dtype=F64, requires_grad=True) for _ in range(2))

    def moved(T, xi):
        rho, phi = xi[0:3], xi[3:6]
        zero = torch.zeros_like(phi[0])
        hat = torch.stack([torch.stack([zero, -phi[2], phi[1]]), torch.stack([phi[2], zero, -phi[0]]),
                           torch.stack([-phi[1], phi[0], zero])])
        return T[:, :3] + hat @ T[:, :3], T[:, 3] + hat @ T[:, 3] + rho

    Ri, ti = moved(Ti, xi_i)
    Rj, tj = moved(Tj, xi_j)
    Y = torch.linalg.solve(Ri, (X - ti).t()).t() @ Rj.t() + tj
    u, v = cam.fx * Y[:, 0] / Y[:, 2] + cam.cx, cam.fy * Y[:, 1] / Y[:, 2] + cam.cy
    x0, y0 = torch.floor(u.detach()), torch.floor(v.detach())
    ok = (Y[:, 2] > 0.2) & (x0 >= 0) & (y0 >= 0) & (x0 + 1 <= W - 1) & (y0 + 1 <= H - 1)
    q = torch.where(ok, y0 * W + x0, torch.zeros_like(x0)).long()
    q = q.clamp(max=W * H - W - 2)
    dd = [Dj.reshape(-1)[q + o] for o in (0, 1, W, W + 1)]
    ww = [w.reshape(-1)[q + o] for o in (0, 1, W, W + 1)]
    ok &= (dd[0] > 0) & (dd[1] > 0) & (dd[2] > 0) & (dd[3] > 0)
    fu, fv = u - x0, v - y0
    a = [(1 - fu) * (1 - fv), fu * (1 - fv), (1 - fu) * fv, fu * fv]
    r = sum(p * t for p, t in zip(a, ww)) * (sum(p * t for p, t in zip(a, dd)) - Y[:, 2])
    huber = torch.where(r.abs() <= 0.05, 0.5 * r * r, 0.05 * (r.abs() - 0.025))
    loss = 300.0 * torch.where(ok, huber, torch.zeros_like(huber)).sum()
    loss.backward()
    return torch.cat([loss.detach().reshape(1), xi_i.grad, xi_j.grad])


def exact(case, seed):
    if case["kind"] == "track":
        # a hundred steps of the sign of a gradient near the minimum amplify the
        # last bit of every sum: the trajectory has no 64-bit value to be held to
        return None
    s = _inputs(case, seed)
    return {"splat": _exact_splat, "render": _exact_render, "mapping": _exact_mapping, "lm": _exact_lm,
            "infer": _exact_infer, "train": _exact_train, "mp": _exact_mp, "keyframe": _exact_keyframe}[case["kind"]](s)
