"""The work that users of this framework have it do, as cases that can be timed.

Every case goes through the package's public entry points on seeded synthetic
RGB-D frames (the package's scene generator: Kinect-like depth noise and
dropout, HD colour).  Volume and image sizes are those of the repository's
workloads, or lie between them.

  static    a geometry-only scanner that owns its volume: one frame fused into
            caller-owned linear arrays per pass
  fuse      a scan: a burst of frames fused into both volumes, which are then
            read out into device tensors.  resume: every pass starts from a
            checkpoint held on the device (a scan taken up again, its free
            space not yet saturated); otherwise the volumes stay as they are
            from pass to pass (a long scan, where most voxels have reached
            their weight limit)
  batch     many independent scans of uneven size, one graph launch per step,
            then all of them read out
  adjoint   calibration refinement: fused colours, their photometric loss and
            its gradients (HD images, intrinsics, extrinsic)
  raycast   a view of the fused volumes (range, vertices, normals, colours)
  track     the pose of a new depth frame against the fused volume
  export    mesh and texture maps of a finished scan
  live      the whole scanning loop for one camera frame in host memory: track
            it, fuse it at the tracked pose, draw the volumes from there
"""
import math

import numpy as np
import torch

import paper_1602_06645_gb300 as T
from paper_1602_06645_gb300 import synth
from paper_1602_06645_gb300.adjoint import Adjoint, fuse_colours

MAX_WEIGHT = 64


def listed():
    return [
        # the smallest call: a 128^3 geometry volume of the caller's, one Kinect frame
        dict(name="static_128", kind="static", gx=128, gy=128, gz=128, extent=1.0, before=3),
        # the small fusion workload: 128^3 / 256^3 over a 1 m cube, 10 frames, a long scan
        dict(name="fuse_small_128_256", kind="fuse", scene="small", gx=128, gy=128, gz=128, num=2, den=1, extent=1.0,
             before=0, frames=10, rgb=1080, colour_mode=0, sample_mode=0, resume=False, ready=True),
        # the scan workload: 512^3 / 1024^3 over a 2 m cube, taken up after 5 frames for 20 more
        dict(name="fuse_scan_512_1024", kind="fuse", scene="scan", gx=512, gy=512, gz=512, num=2, den=1, extent=2.0,
             before=5, frames=20, rgb=1080, colour_mode=0, sample_mode=0, resume=True, ready=True),
        # the asymmetry sweep's ratio 3 on a volume that is no multiple of the brick size, with the paper's
        # normal-weighted colours and bilinear HD samples, frames ordered after the caller's stream
        dict(name="fuse_ratio3_ragged", kind="fuse", scene="sweep", gx=250, gy=243, gz=229, num=3, den=1, extent=1.0,
             before=4, frames=10, rgb=1080, colour_mode=1, sample_mode=1, resume=True, ready=False),
        # the batched workload: scans with log-uniform edges 64..384 and 720p colour
        dict(name="batch_12", kind="batch", scans=12, edges=110, low=64, high=384, steps=6),
        # calibration refinement at 256^3 / 512^3 with 20 full-HD frames
        dict(name="adjoint_256_512", kind="adjoint", gx=256, num=2, frames=20, rgb=1080),
        # a depth-camera view of the scan volumes
        dict(name="raycast_scan", kind="raycast", gx=512, num=2, extent=2.0, before=24, width=640, height=480),
        # a full-HD view (the colour camera's) of a small scan
        dict(name="raycast_hd", kind="raycast", gx=192, num=2, extent=2.0, before=16, width=1920, height=1080),
        # tracking a Kinect frame in the scan volumes
        dict(name="track_scan", kind="track", gx=512, num=1, extent=2.0, before=24, levels=3),
        # mesh and texture maps of the finished scan
        dict(name="export_scan", kind="export", gx=512, num=2, extent=2.0, before=24),
        # the scanning loop at 256^3 / 512^3, frames in page-locked host memory
        dict(name="live_256_512", kind="live", gx=256, num=2, extent=1.0, frames=8, rgb=1080),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["static", "fuse", "fuse", "batch", "adjoint", "raycast", "raycast", "track", "export", "live"])
    if kind == "static":
        return dict(kind=kind, gx=size(40, 320), gy=size(40, 320), gz=size(40, 320), extent=1.0, before=rng.randint(0, 4))
    if kind == "fuse":
        num, den = rng.choice([(1, 1), (2, 1), (3, 1), (5, 3)])
        edge = size(64, 320 if num < 3 else 256)
        g = [max(den, (edge - rng.choice([0, 0, rng.randint(0, edge // 5)])) // den * den) for _ in range(3)]
        return dict(kind=kind, scene=rng.choice(["small", "sweep", "scan"]), gx=g[0], gy=g[1], gz=g[2], num=num, den=den,
                    extent=rng.choice([1.0, 2.0]), before=rng.randint(1, 6), frames=size(2, 16),
                    rgb=rng.choice([720, 1080]), colour_mode=rng.randint(0, 1), sample_mode=rng.randint(0, 1),
                    resume=rng.random() < 0.5, ready=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind=kind, scans=size(2, 16), edges=rng.randint(0, 9999), low=64, high=size(96, 224),
                    steps=rng.randint(1, 4))
    if kind == "adjoint":
        return dict(kind=kind, gx=size(64, 256), num=rng.choice([1, 2]), frames=size(3, 20), rgb=rng.choice([720, 1080]))
    if kind == "raycast":
        return dict(kind=kind, gx=size(64, 448), num=rng.choice([1, 2]), extent=rng.choice([1.0, 2.0]),
                    before=rng.randint(4, 20), width=size(160, 1920), height=size(120, 1080))
    if kind == "track":
        return dict(kind=kind, gx=size(96, 448), num=1, extent=rng.choice([1.0, 2.0]), before=rng.randint(6, 20),
                    levels=rng.randint(1, 3))
    if kind == "export":
        return dict(kind=kind, gx=size(64, 448), num=rng.choice([1, 2]), extent=rng.choice([1.0, 2.0]),
                    before=rng.randint(4, 20))
    return dict(kind=kind, gx=size(96, 320), num=rng.choice([1, 2]), extent=1.0, frames=size(4, 12),
                rgb=rng.choice([720, 1080]))


# ---------------------------------------------------------------- inputs ----
def _spin(seed, salt=0):
    """A number in [0, 1) from the seed."""
    return (synth.splitmix64(seed * 7 + salt) >> 11) / float(1 << 53)


class _Scene:
    """A seeded scene in a cube of side `extent` and its camera path."""

    def __init__(self, kind, extent, n, step_deg, seed, rgb=1080):
        if kind == "scan":
            self.scene = synth.scene_random_primitives(seed, 20 if extent > 1.5 else 5, extent)
        else:
            self.scene = synth.scene_sphere_box_plane(seed) if kind == "small" else synth.scene_plane_sphere(seed)
        self.seed = seed
        self.poses = synth.orbit_poses(n, 0.8 * extent, 25.0, step_deg, target=(0.0, 0.0, -0.15 * extent / 2 - 0.05),
                                       elev_amp_deg=8.0, jitter_t=1e-3, jitter_deg=0.1, seed=seed,
                                       phase_deg=360.0 * _spin(seed))
        self.Kd = synth.K_DEPTH
        self.Kr, self.csz = (synth.K_RGB_1080, synth.RGB_1080) if rgb == 1080 else (synth.K_RGB_720, synth.RGB_720)
        self.Tdr = synth.rig_depth_to_rgb()

    def depth(self, f):
        return synth.render_depth(self.scene, self.Kd, self.poses[f], seed=self.seed, frame=f)

    def rgb(self, f):
        return synth.render_rgb(self.scene, self.Kr, synth.rgb_pose(self.poses[f], self.Tdr), self.csz)

    def args(self, f):
        return self.Kd, self.Kr, self.poses[f], self.Tdr


def _dev(a):
    return torch.from_numpy(a.view(np.int16) if a.dtype == np.uint16 else a).cuda()


def _pinned(a):
    return torch.from_numpy(a.view(np.int16) if a.dtype == np.uint16 else a).pin_memory()


def _grid(case):
    """(geometry dims, colour dims, voxel size, mu)."""
    g = (case["gx"], case.get("gy", case["gx"]), case.get("gz", case["gx"]))
    c = tuple(n * case.get("num", 1) // case.get("den", 1) for n in g)
    vs = float(np.float32(case.get("extent", 1.0) / max(g)))
    return g, c, vs, float(np.float32(3 * vs))


def _volume(case, **kw):
    g, c, vs, mu = _grid(case)
    return T.Volume(g, c, vs, mu, MAX_WEIGHT, **kw)


def _scene_of(case, seed):
    kind = case["kind"]
    if kind == "static":
        return _Scene("small", case["extent"], case["before"] + 1, 9.0, seed)
    if kind == "fuse":
        step = {"scan": 1.2, "small": 36.0, "sweep": 3.6}[case["scene"]]
        return _Scene(case["scene"], case["extent"], case["before"] + case["frames"], step, seed, case["rgb"])
    if kind == "adjoint":
        return _Scene("small", 1.0, case["frames"], 18.0, seed, case["rgb"])
    if kind == "live":
        return _Scene("small", case["extent"], case["frames"], 1.2, seed, case["rgb"])
    # views of a finished scan: frames around the whole orbit, then one more a little further on
    s = _Scene("scan", case["extent"], case["before"], 360.0 / case["before"], seed, 720)
    extra = _Scene("scan", case["extent"], 2, 1.2, seed, 720)
    s.view = extra.poses[1]
    return s


def _edges(case):
    rng = synth.Counter(case["edges"])
    lo, hi = math.log(case["low"]), math.log(case["high"])
    return [int(8 * round(math.exp(rng.uniform(lo, hi)) / 8)) for _ in range(case["scans"])]


def _batch_grid(edge):
    return dict(gx=edge, num=2, extent=1.0)


def _batch_scene(case, seed, i):
    return _Scene("scan", 1.0, case["steps"] + 1, 12.0, seed * 64 + i, 720)


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind == "batch":
        scenes = [_batch_scene(case, seed, i) for i in range(case["scans"])]
        state["vols"] = [_volume(_batch_grid(e)) for e in _edges(case)]
        state["steps"] = [[(_dev(s.depth(f)), _dev(s.rgb(f))) + s.args(f) for s in scenes]
                          for f in range(case["steps"] + 1)]
        torch.cuda.synchronize()
        state["batch"] = T.Batch(state["vols"])
        state["batch"].integrate(state["steps"].pop(0))
        return state
    s = _scene_of(case, seed)
    state["scene"] = s
    if kind == "static":
        g, _, vs, mu = _grid(case)
        state["F"] = torch.zeros(g[::-1], dtype=torch.float32, device="cuda")
        state["W"] = torch.zeros(g[::-1], dtype=torch.uint8, device="cuda")
        state["depth"] = [_dev(s.depth(f)) for f in range(case["before"] + 1)]
        for f in range(case["before"]):
            _static(state, f)
        return state
    if kind == "adjoint":
        state["vol"] = vol = _volume(dict(case, extent=1.0))
        adj = state["adj"] = Adjoint(vol, case["frames"])
        for f in range(case["frames"]):
            adj.record(s.depth(f), s.Kd, s.poses[f])
        adj.finalize()
        state["order"] = torch.argsort(adj.voxels)
        state["target"] = _target(adj.voxels, vol.dims_col)
        state["images"] = torch.stack([_dev(s.rgb(f)) for f in range(case["frames"])]).float().requires_grad_()
        K = s.Kr
        state["K4"] = torch.tensor([K[0, 0], K[1, 1], K[0, 2], K[1, 2]], dtype=torch.float32,
                                   requires_grad=True)
        state["xi"] = torch.zeros(6, dtype=torch.float64, requires_grad=True)
        state["T0"] = _start_extrinsic(s)
        return state
    if kind == "live":
        vol = state["vol"] = _volume(case)
        n = case["frames"]
        state["frames"] = [(_pinned(s.depth(f)), _pinned(s.rgb(f))) for f in range(n)]
        for f in range(n):
            vol.integrate(*state["frames"][f], *s.args(f))
        vol.synchronize()
        state["at"], state["pose"] = 0, np.asarray(s.poses[0], np.float64)
        return state
    if kind == "fuse":
        vol = state["vol"] = _volume(case, colour_mode=case["colour_mode"], sample_mode=case["sample_mode"],
                                     device_inputs_ready=case["ready"])
        for f in range(case["before"]):
            vol.integrate(s.depth(f), s.rgb(f), *s.args(f))
        if case["resume"]:
            state["checkpoint"] = vol.read_torch()
        state["frames"] = [(_dev(s.depth(f)), _dev(s.rgb(f))) + s.args(f)
                           for f in range(case["before"], case["before"] + case["frames"])]
        torch.cuda.synchronize()
        return state
    vol = state["vol"] = _volume(case)
    for f in range(case["before"]):
        vol.integrate(s.depth(f), s.rgb(f), *s.args(f))
    vol.synchronize()
    if kind == "raycast":
        w, h = case["width"], case["height"]
        state["K"] = _view_K(w, h)
    if kind == "track":
        state["depth"] = _dev(synth.render_depth(s.scene, s.Kd, s.view, seed=seed, frame=1000))
        p = state["params"] = T.tsdf_track_params_default()
        p.levels = case["levels"]
        state["params"].far_m = 6.0 if case["extent"] > 1.5 else 4.0
    return state


def _view_K(w, h):
    """A camera with the depth camera's field of view and w x h pixels."""
    f = 525.0 * w / 640.0
    return synth.intrinsics(f, f, (w - 1) / 2.0, (h - 1) / 2.0)


def _start_extrinsic(s):
    """The rig's extrinsic, off by half a degree and 5 mm: where a refinement starts."""
    D = np.eye(4)
    D[:3, :3] = synth.rot_axis_angle((0.3, 0.9, -0.2), math.radians(0.5))
    D[:3, 3] = (0.003, -0.004, 0.001)
    return (D @ np.asarray(s.Tdr, np.float64)).astype(np.float32)


def _target(voxels, dims):
    """Smooth target colours of colour voxels (linear indices)."""
    v = voxels.long() & 0xFFFFFFFF
    x, y, z = v % dims[0], (v // dims[0]) % dims[1], v // (dims[0] * dims[1])
    k = 6.0 / dims[0]
    return torch.stack([128 + 100 * torch.sin(k * x.float()), 128 + 100 * torch.cos(k * y.float()),
                        128 + 100 * torch.sin(k * z.float() + 1.0)], dim=1)


# ------------------------------------------------------------------- run ----
def _static(state, f):
    g, _, vs, mu = _grid(state["case"])
    origin = [-0.5 * n * vs for n in g]
    T.tsdf_integrate_geometry_static(g, vs, mu, MAX_WEIGHT, origin, state["F"], state["W"], state["depth"][f],
                                     state["scene"].Kd, state["scene"].poses[f],
                                     torch.cuda.current_stream().cuda_stream)


_HASH = None


def _canonical(tri):
    """Triangles come in no fixed order: put them in one that depends on their values only."""
    global _HASH
    if _HASH is None:
        _HASH = torch.tensor([synth.splitmix64(i) // 2 | 1 for i in range(9)], dtype=torch.int64, device="cuda")
    key = (tri.reshape(-1, 9).view(torch.int32).long() * _HASH).sum(1)
    return tri[torch.argsort(key)]


def _padded(x, rows):
    """x in a buffer of a size that does not depend on how much was found, zeros after it."""
    out = x.new_zeros((rows,) + tuple(x.shape[1:]))
    out[:len(x)] = x[:rows]
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "static":
        _static(state, case["before"])
        return {"F": state["F"], "W": state["W"]}
    if kind == "fuse":
        vol = state["vol"]
        if case["resume"]:
            vol.write(*state["checkpoint"])
        for fr in state["frames"]:
            vol.integrate(*fr)
        F, W, C = vol.read_torch()
        return {"F": F, "W": W, "C": C}
    if kind == "batch":
        for frames in state["steps"]:
            state["batch"].integrate(frames)
        return [dict(zip("FWC", v.read_torch())) for v in state["vols"]]
    if kind == "adjoint":
        C, n = fuse_colours(state["images"], state["K4"], state["xi"], state["adj"], state["T0"])
        loss = ((C - state["target"]) ** 2).sum()
        gI, gK, gxi = torch.autograd.grad(loss, (state["images"], state["K4"], state["xi"]))
        order, rows = state["order"], 24 * case["gx"] ** 2
        return {"C": _padded(C.detach()[order], rows), "n": _padded(n[order], rows), "gI": gI, "gK": gK, "gxi": gxi}
    if kind == "raycast":
        return state["vol"].raycast(state["K"], state["scene"].view, (case["width"], case["height"]), far=6.0,
                                    device="cuda")
    if kind == "track":
        s = state["scene"]
        pose, rep = T.tsdf_track(state["vol"].h, state["depth"], s.Kd, s.poses[0], np.asarray(s.poses[0], np.float64),
                                 state["params"])
        k = rep.steps
        return {"pose": pose, "A": np.array(rep.A)[:k], "g": np.array(rep.g)[:k], "err2": np.array(rep.err2)[:k],
                "pairs": np.array(rep.correspondences)[:k]}
    if kind == "export":
        vol = state["vol"]
        tri = _canonical(vol.mesh(device="cuda"))
        wh, off, texels = vol.texture_maps(tri, vol.info().voxel_col)
        rows = 6 * case["gx"] ** 2
        return {"triangles": _padded(tri, rows), "wh": _padded(wh, rows), "offsets": _padded(off, rows),
                "texels": _padded(texels, 8 * rows)}
    # live: there and back along the camera path
    s, n = state["scene"], case["frames"]
    k = state["at"] % (2 * n - 2) if n > 1 else 0
    f = k if k < n else 2 * n - 2 - k
    if f == 0:  # the scan's first frame defines the world
        state["pose"] = np.asarray(s.poses[0], np.float64)
    state["at"] += 1
    depth, rgb = state["frames"][f]
    pose, _ = T.tsdf_track(state["vol"].h, depth, s.Kd, state["pose"].astype(np.float32), state["pose"], report=False)
    state["pose"] = pose
    p32 = _rigid32(pose)
    state["vol"].integrate(depth, rgb, s.Kd, s.Kr, p32, s.Tdr)
    out = state["vol"].raycast(s.Kd, p32, synth.DEPTH_SIZE, device="cuda")
    out["pose"] = pose
    return out


def _rigid32(pose):
    """The pose in binary32 with its last row as given."""
    p = pose.astype(np.float32)
    p[3] = (0.0, 0.0, 0.0, 1.0)
    return p


# ------------------------------------------------------------------ work ----
def work(case):
    kind = case["kind"]
    depth = 640 * 480 * 2
    px = {1080: 1920 * 1080, 720: 1280 * 720}[case.get("rgb", 720)]
    if kind == "batch":
        vox = [e ** 3 for e in _edges(case)]
        n = len(vox) * case["steps"]
        return {"bytes": n * (depth + 1280 * 720 * 3) + sum(2 * (5 * v + 32 * v) for v in vox),
                "flops": sum(0.2 * v * 40 for v in vox) * case["steps"]}
    g, c, _, _ = _grid(case)
    ng, nc = g[0] * g[1] * g[2], c[0] * c[1] * c[2]
    if kind == "static":  # F and w of the caller's volume, one depth image
        return {"bytes": depth + 10 * ng, "flops": 40 * 0.5 * ng}
    if kind == "fuse":  # the frames, the volumes before and after
        return {"bytes": case["frames"] * (depth + 3 * px) + 2 * (5 * ng + 4 * nc), "flops": case["frames"] * 40 * 0.2 * ng}
    if kind == "adjoint":  # the images, read in each direction, and their gradient
        return {"bytes": case["frames"] * px * 12 * 3, "flops": case["frames"] * 6.0 * g[0] ** 2 * 400}
    if kind == "raycast":  # four maps, and the cell, colour and normal cells of each hit
        n = case["width"] * case["height"]
        return {"bytes": n * (32 + 40 * 7 + 4), "flops": n * 100 * 30}
    if kind == "track":  # the depth image and, per level, the prediction and each step's maps
        n = 640 * 480
        steps = {1: 10.0, 2: 11.25, 3: 11.5}[case["levels"]]
        return {"bytes": depth + n * 40 * 7 + n * 48 * steps, "flops": n * (100 * 30 + 150 * steps)}
    if kind == "export":  # the observed shell of the volumes, triangles and texels out
        shell = 5.0 * g[0] ** 2
        return {"bytes": shell * 4 * (5 + 4 * case["num"] ** 3) + shell * (36 + 4 * 6), "flops": shell * 500}
    n = 640 * 480
    return {"bytes": depth + 3 * px + 2 * n * (32 + 40 * 7) + n * 48 * 11.5, "flops": 2 * n * 100 * 30 + 40 * 0.1 * ng}


# ----------------------------------------------------------------- exact ----
F64 = torch.float64


def _m64(a):
    return torch.tensor(np.asarray(a, np.float64), dtype=F64, device="cuda")


def _axis64(n, vs):
    """Voxel centres along an axis of n voxels of a cube centred on the origin."""
    o = float(np.float32(-0.5 * n * vs))
    return o + (torch.arange(n, dtype=F64, device="cuda") + 0.5) * vs


def _to_camera(pose, X, Y, Z):
    R, t = _m64(pose)[:3, :3], _m64(pose)[:3, 3]
    X, Y, Z = X - t[0], Y - t[1], Z - t[2]
    return [R[0, i] * X + R[1, i] * Y + R[2, i] * Z for i in range(3)]


def _pixel(K, P, w, h):
    """(nearest pixel index, inside) of camera points."""
    K = np.asarray(K, np.float64)
    u, v = torch.floor(K[0, 0] * P[0] / P[2] + K[0, 2] + 0.5), torch.floor(K[1, 1] * P[1] / P[2] + K[1, 2] + 0.5)
    ok = (P[2] > 0) & (u >= 0) & (u < w) & (v >= 0) & (v < h)
    return torch.where(ok, v * w + u, torch.zeros_like(u)).long(), ok


def _depth64(d):
    return torch.from_numpy(d.astype(np.float64)).cuda() * 0.001


def _update64(F, W, depth, K, pose, g, vs, mu, max_weight=MAX_WEIGHT):
    """The weighted running average of the truncated projective distance, in 64 bits."""
    h, w = depth.shape
    ax = [_axis64(n, vs) for n in g]
    step = max(1, (1 << 24) // (g[0] * g[1]))
    for z0 in range(0, g[2], step):
        z1 = min(g[2], z0 + step)
        P = _to_camera(pose, ax[0][None, None, :], ax[1][None, :, None], ax[2][z0:z1, None, None])
        at, ok = _pixel(K, P, w, h)
        d = depth.reshape(-1)[at]
        sdf = d - P[2]
        up = ok & (d > 0) & (sdf >= -mu)
        t = torch.clamp(sdf / mu, max=1.0)
        f, n = F[z0:z1], W[z0:z1]
        F[z0:z1] = torch.where(up, (f * n + t) / (n + 1), f)
        W[z0:z1] = torch.where(up, torch.clamp(n + 1, max=max_weight), n)


def _fused64(scene, frames, g, vs, mu):
    F = torch.zeros(g[::-1], dtype=F64, device="cuda")
    W = torch.zeros(g[::-1], dtype=F64, device="cuda")
    for f in frames:
        _update64(F, W, _depth64(scene.depth(f)), scene.Kd, scene.poses[f], g, vs, mu)
    return F, W


def _trilinear64(F, W, g, vs, p):
    """(value, exists) of the trilinear distance at points p (n, 3)."""
    i0, fr, ok = [], [], torch.ones(len(p), dtype=torch.bool, device="cuda")
    for a in range(3):
        q = (p[:, a] - float(np.float32(-0.5 * g[a] * vs))) / vs - 0.5
        fl = torch.floor(q)
        ok &= (fl >= 0) & (fl + 1 <= g[a] - 1)
        i0.append(torch.clamp(fl, 0, max(g[a] - 2, 0)).long())
        fr.append(q - fl)
    val = torch.zeros(len(p), dtype=F64, device="cuda")
    for k in range(8):
        o = [k & 1, (k >> 1) & 1, k >> 2]
        at = ((i0[2] + o[2]) * g[1] + i0[1] + o[1]) * g[0] + i0[0] + o[0]
        ok &= W.reshape(-1)[at] > 0
        wgt = 1.0
        for a in range(3):
            wgt = wgt * (fr[a] if o[a] else 1 - fr[a])
        val += wgt * F.reshape(-1)[at]
    return val, ok


def _raycast64(F, W, g, vs, mu, K, pose, w, h, near, far):
    """First + to - crossing along each ray, steps of half a voxel inside the band and mu / 2 elsewhere."""
    K, pose = np.asarray(K, np.float64), _m64(pose)
    n = w * h
    i = torch.arange(n, device="cuda")
    dc = torch.stack([((i % w).to(F64) - K[0, 2]) / K[0, 0], ((i // w).to(F64) - K[1, 2]) / K[1, 1],
                      torch.ones(n, dtype=F64, device="cuda")], 1)
    d = (dc / dc.norm(dim=1, keepdim=True)) @ pose[:3, :3].T
    o = pose[:3, 3]
    rng, normal = torch.zeros(n, dtype=F64, device="cuda"), torch.zeros(n, 3, dtype=F64, device="cuda")
    vertex = torch.zeros(n, 3, dtype=F64, device="cuda")
    live = i
    near, far = float(np.float32(near)), float(np.float32(far))
    t = torch.full((n,), near, dtype=F64, device="cuda")
    tp, Fp = torch.zeros_like(t), torch.zeros_like(t)
    prev = torch.zeros(n, dtype=torch.bool, device="cuda")
    while len(live):
        Fs, ok = _trilinear64(F, W, g, vs, o + t[live, None] * d[live])
        hit = ok & prev[live] & (Fp[live] > 0) & (Fs <= 0)
        at = live[hit]
        rng[at] = tp[at] + (t[at] - tp[at]) * Fp[at] / (Fp[at] - Fs[hit])
        prev[live] = ok
        Fp[live] = torch.where(ok, Fs, Fp[live])
        tp[live] = torch.where(ok, t[live], tp[live])
        t[live] += torch.where(ok & (Fs < 1.0 - 1e-7), 0.5 * vs, 0.5 * mu)
        live = live[~hit]
        live = live[t[live] <= far]
    at = torch.nonzero(rng > 0)[:, 0]
    vertex[at] = o + rng[at, None] * d[at]
    good, gr = torch.ones(len(at), dtype=torch.bool, device="cuda"), []
    for a in range(3):
        e = torch.zeros(3, dtype=F64, device="cuda")
        e[a] = vs
        (fp, o1), (fm, o2) = (_trilinear64(F, W, g, vs, vertex[at] + s * e) for s in (1, -1))
        good &= o1 & o2
        gr.append(fp - fm)
    gr = torch.stack(gr, 1)
    ln = gr.norm(dim=1, keepdim=True)
    normal[at] = torch.where(good[:, None] & (ln > 0), gr / ln, torch.zeros_like(gr))
    return rng, vertex, normal


def _adjoint64(case, s):
    """Gate sets, fused colours, loss and gradients in 64 bits."""
    g, c, vs, mu = _grid(dict(case, extent=1.0))
    sc = g[0] * vs / c[0]
    band = sc / mu
    F = torch.zeros(g[::-1], dtype=F64, device="cuda")
    W = torch.zeros(g[::-1], dtype=F64, device="cuda")
    vox, frame = [], []
    ax = [_axis64(n, sc) for n in c]
    step = max(1, (1 << 23) // (c[0] * c[1]))
    for f in range(case["frames"]):
        depth = _depth64(s.depth(f))
        h, w = depth.shape
        _update64(F, W, depth, s.Kd, s.poses[f], g, vs, mu)
        for z0 in range(0, c[2], step):
            z1 = min(c[2], z0 + step)
            shape = (z1 - z0, c[1], c[0])
            P = _to_camera(s.poses[f], ax[0][None, None, :], ax[1][None, :, None], ax[2][z0:z1, None, None])
            at, ok = _pixel(s.Kd, P, w, h)
            d = depth.reshape(-1)[at]
            ok &= (d > 0) & ((d - P[2]).abs() <= 0.02)
            lin = torch.nonzero(ok.expand(shape).reshape(-1))[:, 0]
            if not len(lin):
                continue
            at, d = at.expand(shape).reshape(-1)[lin], d.expand(shape).reshape(-1)[lin]
            Pq = [q.expand(shape).reshape(-1)[lin] for q in P]
            Kd = np.asarray(s.Kd, np.float64)
            B = [d * ((at % w).to(F64) - Kd[0, 2]) / Kd[0, 0], d * ((at // w).to(F64) - Kd[1, 2]) / Kd[1, 1], d]
            ok = sum((p - b) ** 2 for p, b in zip(Pq, B)) <= float(np.float32(0.02)) ** 2
            lin = lin[ok] + z0 * c[0] * c[1]
            p = torch.stack([ax[0][lin % c[0]], ax[1][(lin // c[0]) % c[1]], ax[2][lin // (c[0] * c[1])]], 1)
            val, ok = _trilinear64(F, W, g, vs, p)
            lin = lin[ok & (val.abs() <= band)]
            vox.append(lin)
            frame.append(torch.full_like(lin, f))
    vox, frame = torch.cat(vox), torch.cat(frame)
    v, slot = torch.unique(vox, return_inverse=True)
    p = torch.stack([ax[0][vox % c[0]], ax[1][(vox // c[0]) % c[1]], ax[2][vox // (c[0] * c[1])]], 1)
    poses = _m64(np.stack(s.poses))[frame]
    P = torch.einsum("nji,nj->ni", poses[:, :3, :3], p - poses[:, :3, 3])
    T0 = _m64(_start_extrinsic(s))
    Q = P @ T0[:3, :3].T + T0[:3, 3]
    K = np.asarray(s.Kr, np.float64)
    images = torch.stack([_dev(s.rgb(f)) for f in range(case["frames"])]).to(F64)
    _, h, w, _ = images.shape
    u, y = K[0, 0] * Q[:, 0] / Q[:, 2] + K[0, 2], K[1, 1] * Q[:, 1] / Q[:, 2] + K[1, 2]
    x0, y0 = torch.floor(u), torch.floor(y)
    ok = (Q[:, 2] > 0) & (x0 >= 0) & (x0 + 1 <= w - 1) & (y0 >= 0) & (y0 + 1 <= h - 1)
    slot_ok, Q, u, y, x0, y0 = slot[ok], Q[ok], u[ok], y[ok], x0[ok], y0[ok]
    a, b = (u - x0)[:, None], (y - y0)[:, None]
    base = (frame[ok] * h + y0.long()) * w + x0.long()
    flat = images.reshape(-1, 3)
    p00, p10, p01, p11 = flat[base], flat[base + 1], flat[base + w], flat[base + w + 1]
    smp = (1 - b) * ((1 - a) * p00 + a * p10) + b * ((1 - a) * p01 + a * p11)
    cnt = torch.zeros(len(v), dtype=F64, device="cuda").index_add_(0, slot_ok, torch.ones_like(u))
    C = torch.zeros(len(v), 3, dtype=F64, device="cuda").index_add_(0, slot_ok, smp) / cnt.clamp(min=1)[:, None]
    gC = 2 * (C - _target(v, c).to(F64))
    gs = gC[slot_ok] / cnt[slot_ok][:, None]
    gI = torch.zeros_like(flat)
    for off, wgt in ((0, (1 - a) * (1 - b)), (1, a * (1 - b)), (w, (1 - a) * b), (w + 1, a * b)):
        gI.index_add_(0, base + off, gs * wgt)
    du = (gs * ((1 - b) * (p10 - p00) + b * (p11 - p01))).sum(1)
    dv = (gs * ((1 - a) * (p01 - p00) + a * (p11 - p10))).sum(1)
    X, Y, Z = Q.T
    gP = torch.stack([du * K[0, 0] / Z, dv * K[1, 1] / Z, -(du * K[0, 0] * X + dv * K[1, 1] * Y) / Z ** 2], 1)
    gK = torch.stack([(du * X / Z).sum(), (dv * Y / Z).sum(), du.sum(), dv.sum()])
    gxi = torch.cat([gP.sum(0), torch.linalg.cross(Q, gP).sum(0)])
    # the rows of C are those of the binary32 gate sets, a few voxels from these: they have no values here
    return {"C": None, "n": None, "gI": gI.reshape(images.shape), "gK": gK.cpu(), "gxi": gxi.cpu()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for i, e in enumerate(_edges(case)):
            g, _, vs, mu = _grid(_batch_grid(e))
            F, _ = _fused64(_batch_scene(case, seed, i), range(case["steps"] + 1), g, vs, mu)
            out.append({"F": F, "W": None, "C": None})
        return out
    # a pose (track, live) is the fixed point of many binary32 decisions, and an export's triangles follow the
    # signs of a fused volume: they have no value of their own in 64 bits
    if kind in ("track", "export", "live"):
        return None
    s = _scene_of(case, seed)
    if kind == "adjoint":
        return _adjoint64(case, s)
    g, c, vs, mu = _grid(case)
    if kind == "static":
        return {"F": _fused64(s, range(case["before"] + 1), g, vs, mu)[0], "W": None}
    if kind == "fuse":
        return {"F": _fused64(s, range(case["before"] + case["frames"]), g, vs, mu)[0], "W": None, "C": None}
    F, W = _fused64(s, range(case["before"]), g, vs, mu)
    w, h = case["width"], case["height"]
    r, v, n = _raycast64(F, W, g, vs, mu, _view_K(w, h), s.view, w, h, 0.1, 6.0)
    return {"range": r.reshape(h, w), "vertex": v.reshape(h, w, 3), "normal": n.reshape(h, w, 3), "rgbw": None}
