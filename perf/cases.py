"""Workloads of the pose search and TSDF fusion library, as a user's program calls them.

A case is a dict of plain values.  `listed()` gives the fixed ones, `draw(rng)` another of the same
ranges, `prepare(case, seed)` builds the inputs and what a program keeps (volume, templates, batch),
`run(state)` makes one pass through the public entry points, `work(case)` counts what a pass cannot do
without and `exact(case, seed)` computes the same outputs in 64 bits with plain torch.

Scene: a room with boxes and spheres inside a cube, seeded; depth images are cast analytically, with
the sensor noise sigma = 0.0012 z^2 and 2% missing pixels.  Volumes hold either the scene's exact
truncated distance (uploaded, for the single operations) or a few fused views of it (for tracking).
"""
import ctypes
import math

import numpy as np
import torch

import paper_2509_24236_gb300 as pf

DTYPES = {"f32": pf.PF_F32, "f16": pf.PF_F16, "bf16": pf.PF_BF16, "fp8": pf.PF_FP8E4M3}
DEV = "cuda"


def listed():
    return [
        # one refinement candidate list on a small map: the smallest call, all launch and set-up time
        dict(name="fitness_few", kind="fitness", w=160, h=120, nx=64, ny=64, nz=64, side=3.2, dtype="f32", view="f32",
             k=64, spread=1.0),
        # first iterations of a full-resolution search, particles degrees and centimetres apart
        dict(name="fitness_spread", kind="fitness", w=640, h=480, nx=512, ny=512, nz=512, side=5.12, dtype="f32",
             view="f32", k=3072, spread=3.0),
        # last iterations of the same search, every particle in nearly the same place
        dict(name="fitness_converged", kind="fitness", w=640, h=480, nx=512, ny=512, nz=512, side=5.12, dtype="f32",
             view="f32", k=3072, spread=0.03),
        # ragged image and grid, particle count off the chunk size, half-precision search view of a float grid
        dict(name="fitness_f16_ragged", kind="fitness", w=317, h=233, nx=251, ny=256, nz=203, side=5.12, dtype="f32",
             view="f16", k=1000, spread=0.3),
        # one frame of the small room: the latency of a whole search on a small map
        dict(name="track_room64", kind="track", w=160, h=120, nx=64, ny=64, nz=64, side=3.2, dtype="f32", view="f32",
             k0=1024, k1=1024, k2=1024, d0=1, d1=1, d2=1, iters=10, update=0),
        # one frame with the paper's schedule of particles and down-sampling: the ordinary call
        dict(name="track_paper", kind="track", w=640, h=480, nx=512, ny=512, nz=512, side=5.12, dtype="f32",
             view="f32", k0=1024, k1=3072, k2=10240, d0=8, d1=16, d2=32, iters=20, update=0),
        # one tracked and fused frame at full resolution, nothing synchronising: the largest call
        dict(name="frame_full", kind="frame", w=640, h=480, nx=512, ny=512, nz=512, side=5.12, dtype="f32",
             view="f32", k0=3072, k1=3072, k2=3072, d0=1, d1=1, d2=1, iters=20, update=0),
        # fusion into the large half-precision map with byte weights, and a small live preview of it
        dict(name="fuse_768_f16", kind="fuse", w=640, h=480, nx=768, ny=768, nz=768, side=6.144, dtype="f16",
             view="f32"),
        # a full-size view of the reconstruction, with normals
        dict(name="raycast_512", kind="raycast", w=640, h=480, nx=512, ny=512, nz=512, side=5.12, dtype="f32",
             view="f32"),
        # training-style use: loss of a batch of frames, gradients of poses and of every voxel
        dict(name="align_grad", kind="align", w=320, h=240, nx=256, ny=256, nz=256, side=5.12, dtype="f32",
             view="f32", frames=64, voxels=True),
        # gradient polish of one frame's pose after its search
        dict(name="polish", kind="polish", w=320, h=240, nx=256, ny=256, nz=256, side=5.12, dtype="f32", view="f32",
             steps=10),
        # twelve sequences of uneven cameras and maps stepped together under one graph, narrow storage
        dict(name="batch_mixed", kind="batch", seqs=12, dtype="bf16", view="f32", kmin=1024, kmax=4096, iters=20,
             scale=1.0),
    ]


def draw(rng):
    """Another case: the kinds of `listed` in turn, sizes spread over their ranges."""
    kind = rng.choice(["fitness", "fitness", "track", "track", "frame", "fuse", "raycast", "align", "polish", "batch"])

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "batch":
        return dict(kind=kind, seqs=rng.randint(2, 10), dtype=rng.choice(["f32", "f16", "bf16", "fp8"]), view="f32",
                    kmin=rng.randint(256, 1024), kmax=rng.randint(1024, 4096), iters=rng.randint(4, 20),
                    scale=round(rng.uniform(0.3, 1.0), 3))
    w = log(120, 640)
    h = max(64, int(w * rng.uniform(0.6, 0.8)))
    big = {"fuse": 768, "raycast": 512, "align": 320, "polish": 320}.get(kind, 512)
    n = log(64, big)
    c = dict(kind=kind, w=w, h=h, nx=n, ny=max(48, n - rng.randint(0, n // 5)), nz=max(48, n - rng.randint(0, n // 5)),
             side=round(rng.uniform(3.2, 6.2), 3), dtype=rng.choice(["f32", "f32", "f16", "bf16", "fp8"]), view="f32")
    if c["dtype"] == "f32" and kind in ("fitness", "track", "frame"):
        c["view"] = rng.choice(["f32", "f32", "f16", "bf16"])
    if kind == "fitness":
        c.update(k=log(16, 4096), spread=round(math.exp(rng.uniform(math.log(0.02), math.log(10.0))), 4))
        c["k"] = min(c["k"], 3072 * 640 * 480 // (w * h))
    elif kind in ("track", "frame"):
        k, d = log(256, 3072), rng.choice([1, 1, 2, 4, 8])
        c.update(k0=k, k1=min(10240, rng.choice([k, 3 * k])), k2=k, d0=d, d1=rng.choice([d, 2 * d]), d2=d,
                 iters=rng.randint(4, 18), update=rng.choice([0, 0, 1]))
        if c["k1"] > k:  # as in the paper's schedule: more particles on fewer points
            c["d1"] = 3 * d
    elif kind == "align":
        c.update(frames=log(1, 64), voxels=rng.random() < 0.7)
        c["w"], c["h"] = min(w, 320), min(h, 240)
    elif kind == "polish":
        c.update(steps=rng.randint(3, 15))
    return c


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------

class _Camera:
    """Pinhole intrinsics of a w x h depth image."""

    def __init__(self, w, h):
        self.width, self.height = w, h
        self.fx = self.fy = float(np.float32(525.0 / 640.0 * w))
        self.cx, self.cy = float(np.float32(0.5 * (w - 1))), float(np.float32(0.5 * (h - 1)))
        self.depth_min, self.depth_max = float(np.float32(0.1)), 8.0


def _geometry(case):
    """(voxel size, truncation) as the library takes them: float32 values."""
    vs = np.float32(case["side"] / max(case["nx"], case["ny"], case["nz"]))
    return float(vs), float(np.float32(3.0) * vs)


def _scene(seed, size):
    """Room interior, boxes at its walls and spheres, as (lo, hi) and (centre, radius), in metres."""
    g = np.random.default_rng(1_000_003 + seed)
    size = np.asarray(size, dtype=np.float64)
    room = (0.06 * size, 0.94 * size)
    boxes, spheres = [], []
    for i in range(6):
        half = size * g.uniform(0.05, 0.10, 3)
        c = size * g.uniform(0.15, 0.85, 3)
        a = i % 3
        c[a] = size[a] * (0.16 if g.random() < 0.5 else 0.84)  # against a wall: the middle stays free
        boxes.append((c - half, c + half))
    for i in range(3):
        r = float(size.min() * g.uniform(0.05, 0.10))
        c = size * np.where(g.random(3) < 0.5, g.uniform(0.15, 0.22, 3), g.uniform(0.78, 0.85, 3))
        spheres.append((c, r))
    return room, boxes, spheres


def _t(v):
    return torch.as_tensor(np.asarray(v), dtype=torch.float64, device=DEV)


def _box_distance(x, lo, hi):
    q = (x - _t(0.5 * (lo + hi))).abs() - _t(0.5 * (hi - lo))
    return q.clamp(min=0.0).norm(dim=-1) + q.max(dim=-1).values.clamp(max=0.0)


def _distance(scene, x):
    room, boxes, spheres = scene
    d = -_box_distance(x, *room)
    for lo, hi in boxes:
        d = torch.minimum(d, _box_distance(x, lo, hi))
    for c, r in spheres:
        d = torch.minimum(d, (x - _t(c)).norm(dim=-1) - r)
    return d


def _analytic_grid(case, seed):
    """(tsdf, weight): the scene's distance over the truncation, clamped; unobserved deep inside matter."""
    vs, trunc = _geometry(case)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    scene = _scene(seed, [vs * (nx - 1), vs * (ny - 1), vs * (nz - 1)])
    i, j = (torch.arange(n, dtype=torch.float64, device=DEV) * vs for n in (nx, ny))
    t = torch.empty((nz, ny, nx), dtype=torch.float32, device=DEV)
    w = torch.empty_like(t)
    for k0 in range(0, nz, 32):
        k = torch.arange(k0, min(nz, k0 + 32), dtype=torch.float64, device=DEV) * vs
        d = _distance(scene, torch.stack(torch.broadcast_tensors(i[None, None, :], j[None, :, None], k[:, None, None]), -1))
        seen = d > -trunc
        t[k0:k0 + 32] = torch.where(seen, (d / trunc).clamp(-1.0, 1.0), torch.ones_like(d)).float()
        w[k0:k0 + 32] = seen.float()
    return t, w


def _rotation(v):
    """exp([v]x) of rotation vectors (..., 3), float64."""
    th = v.norm(dim=-1, keepdim=True).clamp(min=1e-12)[..., None]
    z = torch.zeros_like(v[..., 0])
    k = torch.stack([z, -v[..., 2], v[..., 1], v[..., 2], z, -v[..., 0], -v[..., 1], v[..., 0], z], -1)
    k = k.reshape(v.shape[:-1] + (3, 3)) / th
    eye = torch.eye(3, dtype=torch.float64, device=v.device)
    return eye + torch.sin(th) * k + (1.0 - torch.cos(th)) * (k @ k)


def _pose(R, t):
    P = torch.zeros(R.shape[:-2] + (4, 4), dtype=torch.float64, device=R.device)
    P[..., :3, :3], P[..., :3, 3], P[..., 3, 3] = R, t, 1.0
    return P


def _view(size, seed, turn_deg=0.0, shift=0.0):
    """Camera-to-world pose in the middle of the room, turned and moved a little."""
    g = np.random.default_rng(7_000_003 + seed)
    eye = np.asarray(size) * g.uniform(0.42, 0.58, 3) + shift * g.uniform(-1.0, 1.0, 3)
    # towards a corner and the floor, so that three walls at least hold the pose
    yaw, pitch = math.radians(45.0 + 90.0 * g.integers(4) + g.uniform(-15.0, 15.0) + turn_deg), math.radians(g.uniform(-28.0, -16.0))
    f = np.array([math.cos(pitch) * math.cos(yaw), math.cos(pitch) * math.sin(yaw), math.sin(pitch)])
    r = np.array([math.sin(yaw), -math.cos(yaw), 0.0])
    return _pose(_t(np.stack([r, np.cross(f, r), f], axis=1)), _t(eye))


def _depth(scene, cam, P, gen):
    """Noisy depth image (float32) of the scene from P, 2% of the pixels without a measurement."""
    v, u = torch.meshgrid(torch.arange(cam.height, dtype=torch.float64, device=DEV),
                          torch.arange(cam.width, dtype=torch.float64, device=DEV), indexing="ij")
    d = torch.stack([(u - cam.cx) / cam.fx, (v - cam.cy) / cam.fy, torch.ones_like(u)], -1) @ P[:3, :3].T
    o = P[:3, 3]
    room, boxes, spheres = scene

    def slabs(lo, hi):
        a, b = (_t(lo) - o) / d, (_t(hi) - o) / d
        return torch.minimum(a, b).max(dim=-1).values, torch.maximum(a, b).min(dim=-1).values

    z = slabs(*room)[1]
    for lo, hi in boxes:
        near, far = slabs(lo, hi)
        z = torch.where((near <= far) & (near > 0.0), torch.minimum(z, near), z)
    for c, r in spheres:
        q = o - _t(c)
        a, b, e = (d * d).sum(-1), d @ q, q @ q - r * r
        s = b * b - a * e
        near = (-b - s.clamp(min=0.0).sqrt()) / a
        z = torch.where((s >= 0.0) & (near > 0.0), torch.minimum(z, near), z)
    z = z + 0.0012 * z * z * torch.randn(z.shape, dtype=torch.float64, device=DEV, generator=gen)
    return torch.where(torch.rand(z.shape, device=DEV, generator=gen) < 0.02, torch.zeros_like(z), z).float()


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(99_991 + seed)


def _templates(k, gen):
    t = torch.rand((k, 6), dtype=torch.float32, device=DEV, generator=gen) * 2.0 - 1.0
    t[0] = 0.0
    return t


def _unit(gen):
    v = torch.randn(3, dtype=torch.float64, device=DEV, generator=gen)
    return v / v.norm()


def _perturbation(gen, deg, cm):
    return _pose(_rotation(math.radians(deg) * _unit(gen)), 0.01 * cm * _unit(gen))


def _volume(case, byte_weights=False):
    vs, trunc = _geometry(case)
    return pf.Volume(case["nx"], case["ny"], case["nz"], vs, trunc, tsdf_dtype=DTYPES[case["dtype"]],
                     weight_u8=int(byte_weights), search_dtype=DTYPES[case["view"]])


def _size(case):
    vs, _ = _geometry(case)
    return [vs * (case["nx"] - 1), vs * (case["ny"] - 1), vs * (case["nz"] - 1)]


def _poses(case, P, gen):
    """k float32 3x4 candidates about P: P itself, then moved by up to `spread` degrees and centimetres an axis."""
    u = _templates(case["k"], gen).double()
    R = _rotation(math.radians(case["spread"]) * u[:, :3]) @ P[:3, :3]
    return torch.cat([R, (P[:3, 3] + 0.01 * case["spread"] * u[:, 3:])[..., None]], -1).reshape(-1, 12).float().contiguous()


def _single_frame(case, seed):
    """Camera, pose and depth image of a single operation, and the generator for the rest."""
    cam, gen = _Camera(case["w"], case["h"]), _generator(seed)
    P = _view(_size(case), seed)
    return cam, P, _depth(_scene(seed, _size(case)), cam, P, gen), gen


def _many_frames(case, seed):
    """Poses, perturbed starting poses and points (frames x pixels) of the alignment batch."""
    cam, gen, size = _Camera(case["w"], case["h"]), _generator(seed), _size(case)
    scene = _scene(seed, size)
    truth, starts, depths = [], [], []
    for f in range(case["frames"]):
        P = _view(size, seed, turn_deg=5.0 * f, shift=0.02 * min(size))
        truth.append(P)
        depths.append(_depth(scene, cam, P, gen))
        starts.append(P @ _perturbation(gen, 1.0, 1.0))
    return cam, torch.stack(truth), torch.stack(starts), depths, gen


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _prepare_batch(case, seed)
    if kind == "align":
        cam, _, starts, depths, gen = _many_frames(case, seed)
        s = dict(kind=kind, vol=_volume(case), poses=starts)
        t, w = _analytic_grid(case, seed)
        s["vol"].upload(t.cpu().numpy(), w.cpu().numpy())
        pts = [pf.backproject(d, cam) for d in depths]
        s["points"], s["counts"] = torch.stack([p for p, _ in pts]), torch.cat([n for _, n in pts])
        s["xi"] = (1e-3 * torch.randn((case["frames"], 6), dtype=torch.float64, device=DEV, generator=gen)).requires_grad_()
        n = case["nx"] * case["ny"] * case["nz"]
        s["sink"] = torch.zeros(n, device=DEV, requires_grad=True) if case["voxels"] else None
        return s
    cam, P, depth, gen = _single_frame(case, seed)
    s = dict(kind=kind, cam=cam, depth=depth)
    if kind in ("track", "frame"):
        s["vol"] = _volume(case)
        size, scene = _size(case), _scene(seed, _size(case))
        for turn in (-4.0, 3.0, 0.5):  # what the map holds from earlier frames
            Q = _view(size, seed, turn_deg=turn)
            s["vol"].integrate(_depth(scene, cam, Q, gen), cam, Q.cpu().numpy())
        start = P @ _perturbation(gen, 3.0, 3.0)
        k = [case["k0"], case["k1"], case["k2"]]
        s["params"] = pf.track_params(_templates(max(k), gen), n_iters=case["iters"], k_sched=k,
                                      decim_sched=(case["d0"], case["d1"], case["d2"]), update_mode=case["update"],
                                      compose_mode=1, min_valid_frac=0.05)
        s["vol"].reserve(case["w"] * case["h"], max(k))
        if kind == "track":
            s["start"] = start.cpu().numpy()
        else:
            s["start"], s["pose"] = start.contiguous(), torch.empty((4, 4), dtype=torch.float64, device=DEV)
            s["record"] = torch.zeros(ctypes.sizeof(pf.pf_track_stats), dtype=torch.uint8, device=DEV)
        return s
    s["vol"] = _volume(case, byte_weights=kind == "fuse")
    if kind == "fuse":
        Q = _view(_size(case), seed, turn_deg=6.0)
        s["vol"].integrate(_depth(_scene(seed, _size(case)), cam, Q, gen), cam, Q.cpu().numpy())
        s["pose"] = P.cpu().numpy()
        s["preview"] = _Camera(160, 120)
        return s
    t, w = _analytic_grid(case, seed)
    s["vol"].upload(t.cpu().numpy(), w.cpu().numpy())
    if kind == "raycast":
        s["pose"] = P.cpu().numpy()
        return s
    points, n = pf.backproject(depth, cam)
    points = points[:int(n)].contiguous()
    if kind == "fitness":
        s.update(points=points, poses=_poses(case, P, gen))
    else:
        s.update(points=points, start=(P @ _perturbation(gen, 0.5, 0.5)).contiguous(), steps=case["steps"])
    return s


def _batch_sequences(case):
    """Width, height, nodes per side and particles of each sequence: cameras and maps of three sizes in turn."""
    cams, grids = ((160, 120), (320, 240), (640, 480)), (128, 256, 384)
    out = []
    for i in range(case["seqs"]):
        (w, h), n = cams[i % 3], grids[(i // 3 + i) % 3]
        f = case["scale"]
        k = case["kmin"] + (case["kmax"] - case["kmin"]) * (i % 4) // 3
        out.append((int(w * f), int(h * f), max(48, int(n * f)), k))
    return out


def _prepare_batch(case, seed):
    gen = _generator(seed)
    vols, cams, params, depths, starts, rels = [], [], [], [], [], []
    for i, (w, h, n, k) in enumerate(_batch_sequences(case)):
        one = dict(nx=n, ny=n, nz=n, side=5.12, dtype=case["dtype"], view=case["view"])
        cam, size = _Camera(w, h), _size(one)
        scene, P = _scene(seed + 31 * i, size), _view(size, seed + 31 * i)
        vol = _volume(one, byte_weights=True)
        for turn in (-4.0, 3.0):
            Q = _view(size, seed + 31 * i, turn_deg=turn)
            vol.integrate(_depth(scene, cam, Q, gen), cam, Q.cpu().numpy())
        vols.append(vol)
        cams.append(cam)
        params.append(pf.track_params(_templates(k, gen), n_iters=case["iters"], k_sched=(k, k, k),
                                      decim_sched=(1, 1, 1), update_mode=0, compose_mode=1, min_valid_frac=0.05))
        depths.append(_depth(scene, cam, P, gen))
        starts.append(P)
        rels.append(_perturbation(gen, 3.0, 3.0))
    batch = pf.Batch(vols, cams, params, use_graph=True)
    batch.set_points_per_block(32768)  # what the tuner takes for this mix
    return dict(kind="batch", batch=batch, iters=case["iters"], depths=depths, rels=rels, starts=starts)


# ---------------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------------

def _record(raw, n):
    """The search record in device memory as tensors, iterations 0 .. n - 1."""
    S, m = pf.pf_track_stats, pf.PF_MAX_ITERS

    def field(name, dtype, count):
        at = getattr(S, name).offset
        return raw[at:at + count * dtype.itemsize].view(dtype)

    out = {q: field(q, torch.float32, m)[:n] for q in ("E0", "E_best", "E_new")}
    out.update({q: field(q, torch.int32, m)[:n] for q in ("best", "n_adv", "n_valid0", "n_eval", "k_used")})
    out["s"], out["poses"] = field("s", torch.float64, 2 * m)[:2 * n], field("pose", torch.float64, 12 * m)[:12 * n]
    return out


def run(s):
    kind, vol = s["kind"], s.get("vol")
    if kind == "fitness":
        E, C = vol.fitness(s["points"], s["poses"])
        return {"fitness": E, "count": C}
    if kind == "track":
        status, pose, record = vol.track_frame(s["depth"], s["cam"], s["params"], s["start"])
        return {"status": status, "pose": pose, "record": record}
    if kind == "frame":
        vol.track_frame_async(s["depth"], s["cam"], s["params"], s["start"], s["pose"], s["record"])
        vol.integrate_async(s["depth"], s["cam"], s["pose"])
        return {"pose": s["pose"], "record": _record(s["record"], s["params"].n_iters)}
    if kind == "fuse":
        # the map itself stays in the library: the preview is what a program sees of it
        vol.integrate(s["depth"], s["cam"], s["pose"])
        depth, normal = vol.raycast(s["preview"], s["pose"])
        return {"depth": depth, "normal": normal}
    if kind == "raycast":
        depth, normal = vol.raycast(s["cam"], s["pose"])
        return {"depth": depth, "normal": normal}
    if kind == "align":
        loss = pf.align_loss(vol, s["points"], s["poses"], s["xi"], counts=s["counts"], tsdf_sink=s["sink"])
        wanted = [s["xi"]] + ([s["sink"]] if s["sink"] is not None else [])
        return {"loss": loss.detach(), "grads": list(torch.autograd.grad(loss.sum(), wanted))}
    if kind == "polish":
        pose = s["start"].clone()
        trace, accepted = vol.polish(s["points"], pose, steps=s["steps"])
        return {"pose": pose, "trace": trace, "accepted": accepted}
    # one step of every sequence: new images and odometry in, then search and fusion
    b = s["batch"]
    for i in range(b.n):
        b.depth[i].copy_(s["depths"][i])
        b.rel[i].copy_(s["rels"][i])
        b.pose[i].copy_(s["starts"][i])
    b.step()
    # copied out: the buffers belong to the batch and go with it
    return {"poses": torch.stack(b.pose), "E": torch.stack([_record(b.stats[i], s["iters"])["E_new"] for i in range(b.n)])}


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------

SAMPLE_FLOPS = 43  # transform 18, fractions 3, seven interpolations 21, sum 1
NODE_BYTES = {"f32": 4, "f16": 2, "bf16": 2, "fp8": 1}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        flops = nbytes = 0
        for w, h, n, k in _batch_sequences(case):
            flops += SAMPLE_FLOPS * w * h * (k + 1) * case["iters"]
            nbytes += w * h * (4 + 8 * NODE_BYTES[case["dtype"]] + 2 * (NODE_BYTES[case["dtype"]] + 1)) + 24 * k
        return {"bytes": nbytes, "flops": flops}
    pixels, node = case["w"] * case["h"], NODE_BYTES[case["dtype"] if case["view"] == "f32" else case["view"]]
    cells = 8 * node * pixels  # the corners of the cell that each point falls in, once
    if kind == "fitness":
        return {"bytes": 16 * pixels + cells + (48 + 8) * case["k"], "flops": SAMPLE_FLOPS * pixels * case["k"]}
    if kind in ("track", "frame"):
        flops = sum(SAMPLE_FLOPS * -(-pixels // case["d%d" % (i % 3)]) * (case["k%d" % (i % 3)] + (case["update"] == 0))
                    for i in range(case["iters"]))
        nbytes = 4 * pixels + cells + 24 * max(case["k0"], case["k1"], case["k2"])
        return {"bytes": nbytes + (_fused_bytes(case) if kind == "frame" else 0), "flops": flops}
    if kind == "fuse":
        return {"bytes": _fused_bytes(case) + 4 * pixels + 160 * 120 * 16, "flops": 40 * _fused_bytes(case) / 6}
    if kind == "raycast":
        _, trunc = _geometry(case)
        samples = pixels * 0.4 * case["side"] / (0.5 * trunc)  # the free path of a ray in steps of half the truncation
        return {"bytes": pixels * 16 + 8 * node * pixels, "flops": 30 * samples}
    if kind == "align":
        nodes = case["nx"] * case["ny"] * case["nz"]
        nbytes = case["frames"] * (16 * pixels + cells) + (4 * nodes if case["voxels"] else 0)
        return {"bytes": nbytes, "flops": case["frames"] * pixels * (2 * 43 + 60 + (40 if case["voxels"] else 0))}
    return {"bytes": 16 * pixels + cells, "flops": (case["steps"] + 1) * pixels * 140}


def _fused_bytes(case):
    """Read and write of the node value and weight of the nodes in front of the camera, up to the surface."""
    vs, _ = _geometry(case)
    z = 0.4 * case["side"]
    nodes = (case["w"] * z / (525.0 / 640.0 * case["w"])) * (case["h"] * z / (525.0 / 640.0 * case["w"])) * z / 3 / vs ** 3
    return 2 * nodes * (NODE_BYTES[case["dtype"]] + (1 if case["kind"] == "fuse" else 4))


# ---------------------------------------------------------------------------------------------
# The same outputs in 64 bits
# ---------------------------------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind == "fitness":
        return _exact_fitness(case, seed)
    if kind == "raycast":
        return _exact_raycast(case, seed)
    if kind == "align":
        return _exact_align(case, seed)
    if kind == "polish":
        return _exact_polish(case, seed)
    return None  # a search decides by comparing nearly equal sums, and fusion by rounding to pixels


def _stored_grid(case, seed):
    """The uploaded values as the library keeps them: float64, NaN where a node is unobserved, and those
    that the storage rounds to the edge of the band as +-1."""
    t, w = _analytic_grid(case, seed)
    kind = case["dtype"] if case["view"] == "f32" else case["view"]
    if kind == "f16":
        t = t.half()
    elif kind == "bf16":
        t = t.bfloat16()
    elif kind == "fp8":
        t = (t * 256.0).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).float() / 256.0
    t = t.double().clamp(-1.0, 1.0)
    return torch.where(w > 0, t, torch.full_like(t, math.nan))


def _camera_points(depth, cam):
    """Camera-frame points of the usable pixels, rounded as float32 arithmetic rounds them."""
    v, u = torch.meshgrid(torch.arange(cam.height, device=DEV).float(), torch.arange(cam.width, device=DEV).float(), indexing="ij")
    ok = torch.isfinite(depth) & (depth >= cam.depth_min) & (depth <= cam.depth_max)
    f = [torch.tensor(q, dtype=torch.float32, device=DEV) for q in (cam.fx, cam.fy, cam.cx, cam.cy)]
    return torch.stack([(u - f[2]) * depth / f[0], (v - f[3]) * depth / f[1], depth], -1)[ok].double()


def _corners(grid, g):
    """(eight corners (8, ...), fractions (..., 3), lower node, inside) of grid coordinates g (..., 3), x fastest."""
    nz, ny, nx = grid.shape
    top = torch.tensor([nx - 1, ny - 1, nz - 1], dtype=torch.float64, device=DEV)
    c = g.floor()
    ok = ((c >= 0) & (c < top)).all(-1)
    f = g - c
    c = torch.where(ok[..., None], c, torch.zeros_like(c)).long()
    base = c[..., 0] + nx * (c[..., 1] + ny * c[..., 2])
    flat = grid.reshape(-1)
    v = torch.stack([flat[base + o] for o in (0, 1, nx, nx + 1, nx * ny, nx * ny + 1, nx * ny + nx, nx * ny + nx + 1)])
    return v, f, base, ok


def _interpolate(v, f):
    """Trilinear value and its derivative by the grid coordinate."""
    fx, fy, fz = f.unbind(-1)
    dx = v[1::2] - v[0::2]
    x = v[0::2] + fx * dx
    dy = x[1::2] - x[0::2]
    y = x[0::2] + fy * dy
    ddx = dx[0::2] + fy * (dx[1::2] - dx[0::2])
    value = y[0] + fz * (y[1] - y[0])
    return value, torch.stack([ddx[0] + fz * (ddx[1] - ddx[0]), dy[0] + fz * (dy[1] - dy[0]), y[1] - y[0]], -1)


def _residual(grid, g):
    """(value, derivative, lower node, fractions) with value NaN outside the valid cells."""
    v, f, base, ok = _corners(grid, g)
    ok = ok & (v.abs() < 1.0).all(0)
    t, dg = _interpolate(v, f)
    return torch.where(ok, t, torch.full_like(t, math.nan)), dg, base, f


def _exact_fitness(case, seed):
    if case["k"] * case["w"] * case["h"] > 1.0e9:
        return None
    cam, P, depth, gen = _single_frame(case, seed)
    grid, vs = _stored_grid(case, seed), _geometry(case)[0]
    x = _camera_points(depth, cam)
    poses = _poses(case, P, gen).double().reshape(-1, 3, 4)
    out = torch.empty(case["k"], dtype=torch.float64, device=DEV)
    step = max(1, 1_000_000 // x.shape[0])
    for k in range(0, case["k"], step):
        q = poses[k:k + step]
        t = _residual(grid, (x @ q[:, :, :3].mT + q[:, None, :, 3]) / vs)[0].abs()
        ok = t == t
        out[k:k + step] = torch.where(ok, t, torch.zeros_like(t)).sum(-1) / ok.sum(-1)
    out[out != out] = math.inf
    return {"fitness": out, "count": None}


def _exact_raycast(case, seed):
    cam, P, _, _ = _single_frame(case, seed)
    grid, (vs, trunc) = _stored_grid(case, seed), _geometry(case)
    v, u = torch.meshgrid(torch.arange(cam.height, device=DEV).double(), torch.arange(cam.width, device=DEV).double(), indexing="ij")
    d = torch.stack([(u - cam.cx) / cam.fx, (v - cam.cy) / cam.fy, torch.ones_like(u)], -1) @ P[:3, :3].T
    step, hit = 0.5 * trunc, torch.zeros_like(u)
    prev = torch.full_like(u, math.nan)
    for i in range(int((cam.depth_max - cam.depth_min) / step) + 1):
        z = cam.depth_min + i * step
        c, f, _, ok = _corners(grid, (P[:3, 3] + z * d) / vs)
        t = torch.where(ok, _interpolate(c, f)[0], torch.full_like(prev, math.nan))
        new = (hit == 0) & (prev > 0) & (t <= 0)
        hit = torch.where(new, z - step + step * prev / (prev - t), hit)
        prev = t
    return {"depth": hit, "normal": None}


def _left_jacobian(w):
    th2 = (w * w).sum(-1)[..., None, None]
    z = torch.zeros_like(w[..., 0])
    k = torch.stack([z, -w[..., 2], w[..., 1], w[..., 2], z, -w[..., 0], -w[..., 1], w[..., 0], z], -1).reshape(w.shape[:-1] + (3, 3))
    th = th2.sqrt().clamp(min=1e-12)
    a = torch.where(th < 1e-4, 0.5 - th2 / 24, (1 - torch.cos(th)) / th2.clamp(min=1e-24))
    b = torch.where(th < 1e-2, 1 / 6 - th2 / 120 + th2 * th2 / 5040, (th - torch.sin(th)) / (th2 * th).clamp(min=1e-36))
    return torch.eye(3, dtype=torch.float64, device=DEV) + a * k + b * (k @ k)


def _exact_align(case, seed):
    cam, _, starts, depths, gen = _many_frames(case, seed)
    xi = 1e-3 * torch.randn((case["frames"], 6), dtype=torch.float64, device=DEV, generator=gen)
    grid, vs = _stored_grid(case, seed), _geometry(case)[0]
    nz, ny, nx = grid.shape
    losses, gx = [], []
    gv = torch.zeros(nx * ny * nz, dtype=torch.float64, device=DEV)
    R, J = _rotation(xi[:, :3]), _left_jacobian(xi[:, :3])
    for f, d in enumerate(depths):
        y = _camera_points(d, cam) @ (R[f] @ starts[f, :3, :3]).T + R[f] @ starts[f, :3, 3]
        t, dg, base, fr = _residual(grid, (y + xi[f, 3:]) / vs)
        ok = t == t
        t, dg, base, fr, y = t[ok], dg[ok] / vs, base[ok], fr[ok], y[ok]
        losses.append((t * t).sum())
        gx.append(torch.cat([J[f].T @ (2 * t[:, None] * torch.linalg.cross(y, dg)).sum(0), (2 * t[:, None] * dg).sum(0)]))
        if case["voxels"]:
            for c in range(8):
                w = 2 * t
                for a in range(3):
                    w = w * (fr[:, a] if c >> a & 1 else 1 - fr[:, a])
                gv.index_add_(0, base + (c & 1) + nx * (c >> 1 & 1) + nx * ny * (c >> 2), w)
    return {"loss": torch.stack(losses), "grads": [torch.stack(gx)] + ([gv] if case["voxels"] else [])}


def _exact_polish(case, seed):
    cam, P, depth, gen = _single_frame(case, seed)
    T = P @ _perturbation(gen, 0.5, 0.5)
    grid, vs, x = _stored_grid(case, seed), _geometry(case)[0], _camera_points(depth, cam)

    def system(T):
        q = x @ T[:3, :3].T + T[:3, 3]
        t, dg, _, _ = _residual(grid, q / vs)
        ok = t == t
        t, dg, q = t[ok], dg[ok] / vs, q[ok]
        J = torch.cat([torch.linalg.cross(q, dg), dg], -1)
        return J.T @ J, J.T @ t, (t * t).sum() / ok.sum()

    H, b, best = system(T)
    lam, trace = 1e-3, [best]
    for _ in range(case["steps"]):
        d = torch.linalg.solve(H + lam * torch.diag(torch.diag(H)), -b)
        S = _pose(_rotation(d[:3]), d[3:]) @ T
        Hn, bn, got = system(S)
        if got < best:
            H, b, best, T, lam = Hn, bn, got, S, lam / 10
        else:
            lam *= 10
        trace.append(best)
    return {"pose": T, "trace": torch.stack(trace), "accepted": None}
