"""The calls of this library that are timed, their inputs, and what they return in 64 bits.

A case is one call (or one documented sequence of calls) of the Python binding, at a frame size, voxel size and storage form:

* ``track``  one registration against a model (Volume.track), without or with a mask
* ``mask``   the dynamic mask of a frame with a new object (Volume.compute_mask)
* ``frame``  the whole per-frame loop on device buffers (Volume.process)
* ``host``   the same from host buffers (Volume.process_host), as a program fed by a camera driver calls it
* ``vdepth`` virtual depth: a temporary model of n frames, then its ray cast (Volume.reset, integrate, virtual_depth)
* ``batch``  one frame for each of several streams (Batch.process)

Inputs: a camera moving through a 4 x 4 x 3 m room with boxes and spheres, textured at the scale of indoor surfaces, seen with a Kinect-like
noise (axial sigma 0.0012 + 0.0019 (z - 0.4)^2 m, dropout at depth edges, patches without depth).  The model is what the volume holds after
integrating the frames before the one that is passed, at their poses; the registration starts from the previous frame's pose.  The sizes
are those of the repository's configurations: 160x120 at 2 cm, 640x480 at 1 cm, 1280x720 at 0.5 cm (tau 5 cm), and serving streams of
320x240 to 1280x720 at 1 to 4 cm.

Poses are returned as float32: the registration samples, sums and solves in 32 bits, and its 64-bit output only carries the pose (a caller
turns it into float32 to transform points with it).  Masks and filled depths are whole numbers.
"""
import math

import numpy as np
import torch

from paper_1905_02082_gb300 import refusion as R

ROOM_LO, ROOM_HI = (-2.0, -2.0, 0.0), (2.0, 2.0, 3.0)
Z_NEAR, D_MIN, D_MAX = 0.2, 0.2, 5.0
ITERS, STRIDES = (10, 5, 5), (4, 2, 1)
W_C, GAMMA, THETA_PPM, LAMBDA0, EPS, MIN_VALID = 0.025, 0.5, 7000, 1e-4, 1e-6, 10
LUMA = (0.2126, 0.7152, 0.0722)


def _case(name, kind, width, height, voxel_mm, storage="fp32", frames=4, streams=1, mover=False, masked=False):
    return {"name": name, "kind": kind, "width": width, "height": height, "voxel_mm": voxel_mm, "storage": storage, "frames": frames,
            "streams": streams, "mover": mover, "masked": masked}


def listed():
    return [
        # the smallest call: one registration of the tiny configuration, as a robot with a low-resolution depth camera makes it
        _case("track_160x120", "track", 160, 120, 20),
        # the registration alone, the largest part of a frame, at the size of the TUM and Bonn sequences
        _case("track_640x480", "track", 640, 480, 10),
        # the second registration of a frame (masked pixels left out) in the precision form
        _case("track_1280x720_masked_fp16", "track", 1280, 720, 5, "fp16", mover=True, masked=True),
        # dynamics detection alone: a person or object has entered the view
        _case("mask_640x480", "mask", 640, 480, 10, mover=True),
        _case("mask_1280x720_fp16", "mask", 1280, 720, 5, "fp16", mover=True),
        # the whole loop: a small stream, the common RGB-D camera, and the precision form
        _case("frame_320x240", "frame", 320, 240, 20, mover=True),
        _case("frame_640x480", "frame", 640, 480, 10, mover=True),
        _case("frame_1280x720_fp16", "frame", 1280, 720, 5, "fp16", mover=True),
        # the whole loop from host memory, with the mask returned to the host, one call at a time
        _case("host_640x480", "host", 640, 480, 10, mover=True),
        # filling a frame's holes from a temporary model of 10 frames (ten integrations and a ray cast)
        _case("vdepth_640x480", "vdepth", 640, 480, 10, frames=10),
        # a few equal cameras of one machine
        _case("batch_4x640x480", "batch", 640, 480, 10, streams=4, mover=True),
        # a server's batch: 32 streams of mixed sizes (320x240, 640x480, 1280x720) and voxel sizes (1 to 4 cm), every other with a mover
        _case("batch_32_mixed_fp16", "batch", 0, 0, 0, "fp16", streams=32, mover=True),
    ]


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


def draw(rng):
    kind = rng.choice(["track", "track", "mask", "frame", "frame", "host", "vdepth", "batch"])
    storage = rng.choice(["fp32", "fp16"])
    if kind == "batch" and rng.random() < 0.5:
        return _unnamed(_case("", kind, 0, 0, 0, storage, rng.randint(2, 5), rng.randint(2, 24), True))
    width = int(round(math.exp(rng.uniform(math.log(100), math.log(640 if kind == "batch" else 1280)))))
    height = int(round(width * rng.choice([0.5625, 0.6, 0.75])))
    voxel = rng.choice([10, 12, 15, 20, 25, 30, 40]) if kind in ("batch", "vdepth") or width < 320 else rng.choice([5, 8, 10, 12, 15, 20])
    mover = kind in ("mask",) or rng.random() < 0.6
    frames = rng.randint(4, 10) if kind == "vdepth" else rng.randint(2, 6)
    streams = rng.randint(2, 8) if kind == "batch" else 1
    masked = kind == "track" and mover and rng.random() < 0.7
    return _unnamed(_case("", kind, width, height, voxel, storage, frames, streams, mover, masked))


def _streams(case):
    """(width, height, voxel_mm, mover) of each stream."""
    if case["width"]:
        return [(case["width"], case["height"], case["voxel_mm"], case["mover"])] * case["streams"]
    out = []
    for s in range(case["streams"]):
        w, h = ((320, 240), (640, 480), (1280, 720))[s % 3]
        v = (10, 20, 30, 40)[s % 4]
        out.append((w, h, max(v, 20) if w == 1280 else v, case["mover"] and s % 2 == 1))
    return out


def _tau(voxel_mm):
    return 0.05 if voxel_mm < 10 else 0.1


def _intrinsics(w, h):
    """The field of view of 525 pixels of focal length at 640 (the precision camera is the same one, twice as fine)."""
    f = 525.0 * w / 640.0
    return f, f, (w - 1) / 2.0, (h - 1) / 2.0


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

class _Scene:
    def __init__(self, seed):
        g = np.random.default_rng(seed)
        # two boxes and two spheres standing in the corner that the camera looks at, at the range of a desk or a robot's arm
        self.boxes = []
        for _ in range(2):
            half = g.uniform(0.08, 0.2, 3) * np.array([1, 1, 1.6])
            self.boxes.append((np.array([g.uniform(1.25, 1.75), g.uniform(1.25, 1.75), half[2]]), half))
        self.spheres = []
        for _ in range(2):
            r = g.uniform(0.1, 0.25)
            self.spheres.append((np.array([g.uniform(1.2, 1.7), g.uniform(1.2, 1.7), r]), r))
        self.tex = [(g.uniform(14.0, 60.0, 3), g.uniform(0, 6.28, 3), g.uniform(0.35, 0.95, 3)) for _ in range(6)]
        self.eye = np.array([g.uniform(0.45, 0.7), g.uniform(0.45, 0.7), g.uniform(0.9, 1.2)])
        self.target = np.array([1.7, 1.7, 0.4]) + g.uniform(-0.1, 0.1, 3)
        self.step = g.uniform(-1, 1, 3) * np.array([0.008, 0.008, 0.004])
        self.turn = g.uniform(-1, 1, 3) * np.array([0.012, 0.012, 0.01])
        self.mover_at, self.mover_half = g.uniform(0.40, 0.55), np.array([0.1, 0.1, 0.16]) * g.uniform(0.7, 1.2)

    def pose(self, i):
        eye, target = self.eye + i * self.step, self.target + i * self.turn
        z = (target - eye) / np.linalg.norm(target - eye)
        x = np.cross(z, [0.0, 0.0, 1.0])
        x /= np.linalg.norm(x)
        T = np.eye(4)
        T[:3, 0], T[:3, 1], T[:3, 2], T[:3, 3] = x, np.cross(z, x), z, eye
        return T


def _box_t(o, d, c, h):
    a, b = (c - h - o) / d, (c + h - o) / d
    near, far = torch.minimum(a, b).amax(1), torch.maximum(a, b).amin(1)
    return torch.where((near <= far) & (near > 1e-6), near, torch.inf)


def _render(scene, w, h, T, mover, gen):
    """Depth (uint16, mm) and RGB8 of one frame, on the GPU."""
    dev = torch.device("cuda")
    fx, fy, cx, cy = _intrinsics(w, h)
    t64 = lambda v: torch.as_tensor(np.asarray(v, dtype=np.float64), device=dev)  # noqa: E731
    v, u = torch.meshgrid(torch.arange(h, device=dev, dtype=torch.float64), torch.arange(w, device=dev, dtype=torch.float64), indexing="ij")
    dc = torch.stack([(u - cx) / fx, (v - cy) / fy, torch.ones_like(u)], -1).reshape(-1, 3)
    d = dc @ t64(T[:3, :3]).T
    d = torch.where(d.abs() < 1e-12, 1e-12, d)
    o = t64(T[:3, 3])
    t = torch.where(d > 0, (t64(ROOM_HI) - o) / d, (t64(ROOM_LO) - o) / d).amin(1)
    part = torch.zeros_like(t, dtype=torch.long)
    hits = [_box_t(o, d, t64(c), t64(hh)) for c, hh in scene.boxes]
    for c, r in scene.spheres:
        oc, a = o - t64(c), (d * d).sum(1)
        b = (d * oc).sum(1)
        disc = b * b - a * ((oc * oc).sum() - r * r)
        ts = (-b - disc.clamp_min(0).sqrt()) / a
        hits.append(torch.where((disc >= 0) & (ts > 1e-6), ts, torch.inf))
    if mover:
        # an object that the model has not seen: a box between the camera and the room
        T0 = scene.pose(0)
        hits.append(_box_t(o, d, t64(T0[:3, 3] + scene.mover_at * (scene.target - T0[:3, 3])), t64(scene.mover_half)))
    for k, th in enumerate(hits):
        part = torch.where(th < t, k + 1, part)
        t = torch.minimum(t, th)
    p = o + d * t[:, None]
    freq, phase, base = (torch.stack([t64(x[i]) for x in scene.tex])[part] for i in range(3))
    s = torch.sin(freq * p + phase)
    shade = 0.55 + 0.3 * s.prod(1) + 0.15 * torch.sin(freq[:, 0] * p.sum(1) * 0.6 + phase[:, 1])
    rgb = (255.0 * base * shade[:, None] + 2.0 * torch.randn(len(t), 3, device=dev, generator=gen)).clamp(0, 255).round().to(torch.uint8)
    z = t.reshape(h, w)
    # no depth at silhouettes (a band of a few pixels, as structured light leaves it), and patches without depth
    edge = torch.zeros_like(z, dtype=torch.bool)
    for ax in (0, 1):
        jump = torch.diff(z, dim=ax).abs() > 0.03
        n = z.shape[ax]
        edge.narrow(ax, 0, n - 1).logical_or_(jump)
        edge.narrow(ax, 1, n - 1).logical_or_(jump)
    drop = torch.nn.functional.max_pool2d(edge.float()[None, None], 5, 1, 2)[0, 0] > 0
    patches = torch.rand(4, 3, device=dev, generator=gen)
    for a, b, r in patches.cpu().tolist():
        drop |= (u - a * w) ** 2 + (v - b * h) ** 2 < ((0.01 + 0.02 * r) * w) ** 2
    noisy = z + (0.0012 + 0.0019 * (z - 0.4) ** 2) * torch.randn(h, w, device=dev, generator=gen)
    mm = torch.where(drop, 0.0, (1000.0 * noisy).round()).clamp(0, 65535).to(torch.int32).to(torch.uint16)
    return mm.contiguous(), rgb.reshape(h, w, 3).contiguous()


def _sequence(case, seed, stream, frames):
    """The frames of one stream ([(depth, rgb)]), their poses, and the frame that is passed (None for vdepth)."""
    w, h, _, mover = _streams(case)[stream]
    scene = _Scene([int(seed), stream])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 1009 + stream)
    poses = [scene.pose(i) for i in range(frames + 1)]
    model = [_render(scene, w, h, poses[i], False, gen) for i in range(frames)]
    now = None if case["kind"] == "vdepth" else _render(scene, w, h, poses[frames], mover, gen)
    return model, poses, now


def _blocks(voxel_mm):
    """Pool and bucket count for a whole room at this voxel size, with room to spare."""
    n = int(1.6 * 4.4 * 4.4 * 3.4 / (8e-3 * voxel_mm) ** 3) + 2000
    return n, 1 << max(12, (n - 1).bit_length())


def _volume(case, stream, model, poses):
    w, h, voxel, _ = _streams(case)[stream]
    n, buckets = _blocks(voxel)
    vol = R.Volume(n_buckets=buckets, max_blocks=n, max_width=w, max_height=h, voxel_size=voxel * 1e-3, trunc=_tau(voxel),
                   storage=R.STORAGE_FP16 if case["storage"] == "fp16" else R.STORAGE_FP32)
    K = R.Intrinsics(*_intrinsics(w, h))
    for (depth, rgb), T in zip(model, poses):
        vol.integrate(vol.frame(depth, rgb, K), torch.as_tensor(T, device="cuda").contiguous())
    # (Volume.process tracks only once the volume has processed a frame: an empty volume's first frame goes in at its pose)
    return vol, K


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": dict(case)}
    if kind == "vdepth":
        model, poses, _ = _sequence(case, seed, 0, case["frames"])
        w, h, voxel, _ = _streams(case)[0]
        vol, K = _volume(case, 0, [], [])
        s |= {"vol": vol, "keep": model, "frames": [vol.frame(d, c, K) for d, c in model],
              "poses": [torch.as_tensor(T, device="cuda").contiguous() for T in poses], "out": torch.empty(h, w, dtype=torch.uint16, device="cuda")}
        vol.sync()
        return s
    vols, frames, inits, keep = [], [], [], []
    for i in range(case["streams"]):
        model, poses, now = _sequence(case, seed, i, case["frames"])
        loop = kind in ("frame", "host", "batch")
        vol, K = _volume(case, i, [] if loop else model, poses)
        if loop:
            # the first frame through the loop (the volume is empty: integrated at its pose), the others at their poses
            vol.process(vol.frame(*model[0], K), torch.as_tensor(poses[0], device="cuda").contiguous())
            for f, T in zip(model[1:], poses[1:]):
                vol.integrate(vol.frame(*f, K), torch.as_tensor(T, device="cuda").contiguous())
        vols.append(vol)
        frames.append(vol.frame(*now, K))
        inits.append(torch.as_tensor(poses[case["frames"] - 1], device="cuda").contiguous())
        keep.append(now)
        if i == 0:
            s |= {"K": K, "last": poses[case["frames"] - 1], "true": torch.as_tensor(poses[case["frames"]], device="cuda").contiguous()}
        vol.sync()
    w, h, _, _ = _streams(case)[0]
    s |= {"vol": vols[0], "frame": frames[0], "init": inits[0], "keep": keep}
    if kind == "track":
        s["mask"] = vols[0].compute_mask(frames[0], s["true"]) if case["masked"] else None
    elif kind == "host":
        s |= {"depth": keep[0][0].cpu().numpy(), "rgb": keep[0][1].cpu().numpy()}
    elif kind == "batch":
        s |= {"vols": vols, "batch": R.Batch(vols), "frames": frames, "inits": inits,
              "outs": torch.empty(len(vols), 4, 4, dtype=torch.float64, device="cuda"),
              "masks": [torch.empty(a, b, dtype=torch.uint8, device="cuda") for b, a, _, _ in _streams(case)]}
    if kind in ("mask", "frame"):
        s["out"] = torch.empty(h, w, dtype=torch.uint8, device="cuda")
    vols[0].sync()
    return s


def run(s):
    kind, vol = s["case"]["kind"], s["vol"]
    if kind == "track":
        T, _ = vol.track(s["frame"], s["init"], s["mask"])
        return {"pose": T.float()}
    if kind == "mask":
        return {"mask": vol.compute_mask(s["frame"], s["true"], s["out"])}
    if kind == "frame":
        T, _ = vol.process(s["frame"], s["init"], s["out"])
        return {"pose": T.float(), "mask": s["out"]}
    if kind == "host":
        T, mask = vol.process_host(s["depth"], s["rgb"], s["K"], s["last"], want_mask=True)
        return {"pose": T.astype(np.float32), "mask": mask}
    if kind == "vdepth":
        vol.reset()
        for f, T in zip(s["frames"], s["poses"]):
            vol.integrate(f, T)
        return {"depth": vol.virtual_depth(s["frames"][0], s["poses"][0], 0, s["out"])}
    s["batch"].process(s["frames"], s["inits"], list(s["outs"]), s["masks"])
    return {"poses": s["outs"].float(), "masks": s["masks"]}


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------

def work(case):
    """Bytes: each input image, each model voxel that is looked up or updated, and each output once.  The visible surface is taken at 1.4 m
    (the scene's mean depth): three voxel layers of it are looked up, and the voxels in front of it are updated.  Operations: about 320 per
    pixel and cost evaluation, 150 per mask pixel, 60 per updated voxel."""
    total = {"bytes": 0.0, "flops": 0.0}
    fp16 = case["storage"] == "fp16"
    for w, h, voxel, _ in _streams(case):
        px, v = w * h, voxel * 1e-3
        area = px * (1.4 / _intrinsics(w, h)[0]) ** 2
        looked = min(8 * px, 3 * area / v ** 2) * (4 if fp16 else 8)
        updated = area * 1.4 / 3.0 / v ** 3
        reg_flops = sum((n + 1) * (-(-w // st)) * (-(-h // st)) for n, st in zip(ITERS, STRIDES)) * 320.0
        kind, b, f = case["kind"], 0.0, 0.0
        integ_b, integ_f = updated * (8 if fp16 else 18), updated * 60.0
        if kind == "track":
            b, f = 5.0 * px + (px if case["masked"] else 0) + looked + 64, reg_flops
        elif kind == "mask":
            b, f = 3.0 * px + looked, 150.0 * px
        elif kind == "vdepth":
            b, f = case["frames"] * (5.0 * px + integ_b) + 4.0 * px, case["frames"] * integ_f
        else:
            b, f = 6.0 * px + looked + integ_b + 64, 2 * reg_flops + 150.0 * px + integ_f
        total["bytes"] += b
        total["flops"] += f
    return total


# ----------------------------------------------------------------------------
# the same in 64 bits
# ----------------------------------------------------------------------------

class _Grid:
    """The model as dense arrays over the part of the room that the frames see (TSDF, weight, colour, colour weight)."""

    def __init__(self, w, h, voxel, tau, model, poses):
        self.v, self.tau = voxel, tau
        fx, fy, cx, cy = _intrinsics(w, h)
        cam = np.array([[(u - cx) / fx * z, (v - cy) / fy * z, z] for u in (-1, w) for v in (-1, h) for z in (Z_NEAR, D_MAX)])
        pts = np.concatenate([cam @ T[:3, :3].T + T[:3, 3] for T in poses])
        lo = np.maximum(pts.min(0), np.array(ROOM_LO) - tau - 0.15)
        hi = np.minimum(pts.max(0), np.array(ROOM_HI) + tau + 0.15)
        self.lo = np.floor(lo / voxel).astype(int) - 1
        self.n = np.ceil(hi / voxel).astype(int) + 2 - self.lo
        nx, ny, nz = (int(x) for x in self.n)
        F = torch.zeros(nz, ny, nx, dtype=torch.float64, device="cuda")
        W = torch.zeros(nz, ny, nx, dtype=torch.uint8, device="cuda")
        C = torch.zeros(3, nz, ny, nx, dtype=torch.uint8, device="cuda")
        Wc = torch.zeros_like(W)
        ax = [torch.arange(int(n), device="cuda", dtype=torch.float64) * voxel + float(o * voxel) for n, o in zip(self.n, self.lo)]
        slab = max(1, 16_000_000 // (nx * ny))
        for (depth, rgb), T in zip(model, poses):
            D = depth.to(torch.int32).double().reshape(-1) / 1000.0
            ok = (depth.to(torch.int32).reshape(-1) != 0) & (D >= D_MIN) & (D <= D_MAX)
            R3, t = T[:3, :3], T[:3, 3]
            col = rgb.reshape(-1, 3)
            for z0 in range(0, nz, slab):
                z1 = min(nz, z0 + slab)
                dx, dy, dz = ax[0][None, None, :] - t[0], ax[1][None, :, None] - t[1], ax[2][z0:z1, None, None] - t[2]
                c = [float(R3[0, i]) * dx + float(R3[1, i]) * dy + float(R3[2, i]) * dz for i in range(3)]
                inside = (c[2] > Z_NEAR) & (c[2] <= D_MAX)
                at = inside.reshape(-1).nonzero()[:, 0]
                if not len(at):
                    continue
                X, Y, Z = (k.reshape(-1)[at] for k in c)
                u, v = torch.floor(fx * X / Z + cx + 0.5), torch.floor(fy * Y / Z + cy + 0.5)
                keep = (u >= 0) & (u < w) & (v >= 0) & (v < h)
                at, Z = at[keep], Z[keep]
                pix = (v[keep] * w + u[keep]).long()
                sdf = D[pix] - Z
                keep = ok[pix] & (sdf >= -tau)
                at, pix, sdf = at[keep], pix[keep], sdf[keep]
                f, wt = F[z0:z1].reshape(-1), W[z0:z1].reshape(-1)
                wd = wt[at].double()
                f[at] = (wd * f[at] + sdf.clamp_max(tau)) / (wd + 1)
                wt[at] = (wd + 1).clamp_max(255).to(torch.uint8)
                band = sdf <= tau
                at, pix = at[band], pix[band]
                wc = Wc[z0:z1].reshape(-1)
                wd = wc[at].long()
                for k in range(3):
                    ck = C[k, z0:z1].reshape(-1)
                    ck[at] = ((2 * (wd * ck[at].long() + col[pix, k].long()) + wd + 1) // (2 * (wd + 1))).to(torch.uint8)
                wc[at] = (wd + 1).clamp_max(255).to(torch.uint8)
        self.F = torch.where(W > 0, F, torch.nan).reshape(-1)
        del F
        self.C, self.Wc = C.reshape(3, -1), Wc.reshape(-1)

    def at(self, p, colour=True):
        """Value, gradient and validity of the trilinear TSDF, and of the intensity, at world points p [n, 3]."""
        q = p / self.v
        k = torch.floor(q)
        f = (q - k).T
        k = k.long() - torch.as_tensor(self.lo, device=p.device)
        n = torch.as_tensor(self.n, device=p.device)
        inside = ((k >= 0) & (k < n - 1)).all(1)
        k = torch.where(inside[:, None], k, 0)
        nx, ny = int(self.n[0]), int(self.n[1])
        base = (k[:, 2] * ny + k[:, 1]) * nx + k[:, 0]
        idx = [base + (c & 1) + ((c >> 1) & 1) * nx + (c >> 2) * nx * ny for c in range(8)]

        def tri(vals):
            g, val = [0.0, 0.0, 0.0], 0.0
            for c, x in enumerate(vals):
                w = [f[i] if (c >> i) & 1 else 1 - f[i] for i in range(3)]
                s = [1.0 if (c >> i) & 1 else -1.0 for i in range(3)]
                val = val + w[0] * w[1] * w[2] * x
                g[0], g[1], g[2] = g[0] + s[0] * w[1] * w[2] * x, g[1] + s[1] * w[0] * w[2] * x, g[2] + s[2] * w[0] * w[1] * x
            return val, torch.stack(g, 1) / self.v

        V, gV = tri([self.F[i] for i in idx])
        ok = inside & ~torch.isnan(V)
        if not colour:
            return V, ok
        okc = ok.clone()
        for i in idx:
            okc &= self.Wc[i] > 0
        I, gI = tri([sum(LUMA[k] * self.C[k][i].double() for k in range(3)) / 255.0 for i in idx])
        return V, gV, ok, I, gI, okc


def _points(depth, w, h, stride, mask):
    """Camera points of the valid pixels of one sub-sampling, and their indices."""
    fx, fy, cx, cy = _intrinsics(w, h)
    v, u = torch.meshgrid(torch.arange(0, h, stride, device="cuda"), torch.arange(0, w, stride, device="cuda"), indexing="ij")
    idx = (v * w + u).reshape(-1)
    D = depth.to(torch.int32).double().reshape(-1) / 1000.0
    ok = (D[idx] >= D_MIN) & (D[idx] <= D_MAX)
    if mask is not None:
        ok &= mask.reshape(-1)[idx] == 0
    idx = idx[ok]
    z = D[idx]
    return torch.stack([((idx % w).double() - cx) / fx * z, (torch.div(idx, w, rounding_mode="floor").double() - cy) / fy * z, z], 1), idx


def _register(grid, depth, rgb, w, h, T, mask):
    """Levenberg-Marquardt over the three sub-samplings."""
    lum = sum(LUMA[k] * rgb.reshape(-1, 3)[:, k].double() for k in range(3)) / 255.0
    T = torch.as_tensor(T, dtype=torch.float64)
    for n, stride in zip(ITERS, STRIDES):
        x, idx = _points(depth, w, h, stride, mask)

        def cost(T):
            p = x @ T[:3, :3].T.cuda() + T[:3, 3].cuda()
            V, gV, ok, I, gI, okc = grid.at(p)
            J = torch.cat([gV, torch.linalg.cross(p, gV)], 1)[ok]
            r = V[ok]
            Jc = torch.cat([gI, torch.linalg.cross(p, gI)], 1)[okc]
            rc = (I - lum[idx])[okc]
            H = J.T @ J + W_C * (Jc.T @ Jc)
            return H.cpu(), (J.T @ r + W_C * (Jc.T @ rc)).cpu(), float((r * r).sum() + W_C * (rc * rc).sum()), int(ok.sum())

        H, g, E, N = cost(T)
        lam = LAMBDA0
        if N < MIN_VALID:
            continue
        for _ in range(n):
            d = torch.linalg.solve(H + lam * torch.diag(torch.diag(H)), -g)
            if d[:3].norm() < EPS and d[3:].norm() < EPS:
                break
            X = torch.zeros(4, 4, dtype=torch.float64)
            X[0, 1], X[0, 2], X[1, 0], X[1, 2], X[2, 0], X[2, 1] = -d[5], d[4], d[5], -d[3], -d[4], d[3]
            X[:3, 3] = d[:3]
            Tc = torch.linalg.matrix_exp(X) @ T
            Hc, gc, Ec, Nc = cost(Tc)
            if Nc >= MIN_VALID and Ec * N < E * Nc:
                T, H, g, E, N, lam = Tc, Hc, gc, Ec, Nc, lam * 0.1
            else:
                lam *= 10.0
    return T


def _dynamic_mask(grid, depth, w, h, T):
    x, idx = _points(depth, w, h, 1, None)
    V, ok = grid.at(x @ T[:3, :3].T.cuda() + T[:3, 3].cuda(), colour=False)
    V = V.clamp(-grid.tau, grid.tau)
    seeds = torch.zeros(h * w, device="cuda")
    seeds[idx[ok & (V * V > GAMMA * grid.tau ** 2)]] = 1.0
    pool = lambda m: torch.nn.functional.max_pool2d(m[None, None], 3, 1, 1)[0, 0]  # noqa: E731
    pad = torch.ones(h + 2, w + 2, device="cuda")
    pad[1:-1, 1:-1] = 1.0 - seeds.reshape(h, w)
    m = (torch.nn.functional.max_pool2d(pad[None, None], 3, 1)[0, 0] == 0)
    D = depth.to(torch.int64)
    edges = []
    for ax, s in ((0, 1), (0, -1), (1, 1), (1, -1)):
        src = torch.roll(D, s, ax)
        joins = (src - D).abs() * 1_000_000 < THETA_PPM * src
        joins.select(ax, 0 if s == 1 else -1).zero_()
        edges.append((ax, s, joins))
    count = -1
    while int(m.sum()) != count:
        count = int(m.sum())
        for _ in range(16):
            for ax, s, joins in edges:
                m = m | (torch.roll(m, s, ax) & joins)
    return pool(m.float()) > 0


def exact(case, seed):
    """The registered pose of one registration in 32-bit storage.  The others have no such value: masks and filled depths are whole numbers;
    in 16-bit storage the model itself is rounded at every update; and the whole loop registers twice around a mask, 46 accept decisions,
    the last of each level between poses a micrometre apart whose 32-bit mean costs are the same."""
    if case["kind"] != "track" or case["storage"] != "fp32":
        return None
    w, h, voxel, _ = _streams(case)[0]
    model, poses, (depth, rgb) = _sequence(case, seed, 0, case["frames"])
    grid = _Grid(w, h, voxel * 1e-3, _tau(voxel), model, poses)
    last, true = (torch.as_tensor(poses[case["frames"] - k]) for k in (1, 0))
    mask = _dynamic_mask(grid, depth, w, h, true) if case["masked"] else None
    return {"pose": _register(grid, depth, rgb, w, h, last, mask).cuda()}
