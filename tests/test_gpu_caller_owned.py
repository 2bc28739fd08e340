"""The caller-owned geometry volume (tsdf_integrate_geometry_static) against
the oracle where its kernels differ: values that overflow, a volume far from
the world's origin (and the handle's frames there), a depth camera that is no
pinhole (and the handle's frames with one), both forms of the culling on either
side of the line between them, stream capture."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1602_06645_gb300 as T  # noqa: E402
from paper_1602_06645_gb300 import synth  # noqa: E402

K = synth.intrinsics(60.0, 55.0, 39.0, 29.0)
POSES = synth.orbit_poses(3, 0.9, 20.0, 25.0)
# whole bricks; rows of a multiple of four voxels; any other rows
DIMS = [(64, 64, 64), (36, 29, 43), (37, 30, 41)]


def surface(seed, shape=(60, 80)):
    rng = np.random.default_rng(seed)
    d = rng.integers(700, 1100, shape).astype(np.uint16)
    d[rng.random(shape) < 0.05] = 0
    return d


def dev(d):
    return torch.from_numpy(d.view(np.int16)).cuda()


def check(dims, s, F0, W0, frames, Kd, poses, origin=None, max_weight=255):
    """Frames fused into copies of F0 and W0 by the library and by the oracle."""
    org = [-0.5 * m * s for m in dims] if origin is None else origin
    F, W = torch.from_numpy(F0).cuda(), torch.from_numpy(W0).cuda()
    o = oracle.Oracle(dims, dims, s, 3 * s, max_weight, n_threads=8, origin=org)
    o.F[...], o.W[...] = F0, W0
    n = 0
    for d, pose in zip(frames, poses):
        T.tsdf_integrate_geometry_static(dims, s, 3 * s, max_weight, org, F, W, dev(d), Kd, pose)
        n += o.integrate_geometry(d, Kd, pose)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(W.cpu().numpy(), o.W)
    np.testing.assert_array_equal(F.cpu().numpy(), o.F)
    return n


def zeros(dims):
    return np.zeros(dims[::-1], np.float32), np.zeros(dims[::-1], np.uint8)


@pytest.mark.parametrize("dims", DIMS)
def test_values_that_overflow(dims):
    """F of infinite, huge and tiny magnitude and not a number: the average is
    the IEEE fmaf(F, w, t) / (w + 1)."""
    rng = np.random.default_rng(sum(dims))
    odd = np.array([np.inf, -np.inf, np.nan, 3e38, -3e38, 1e-40, -1e-45, 2e-38], np.float32)
    F0 = rng.uniform(-1, 1, dims[::-1]).astype(np.float32)
    F0.reshape(-1)[::3] = rng.choice(odd, F0.reshape(-1)[::3].shape)
    W0 = rng.integers(0, 256, dims[::-1]).astype(np.uint8)
    s = float(np.float32(0.6 / max(dims)))
    assert check(dims, s, F0, W0, [surface(k) for k in range(3)], K, POSES) > F0.size // 20


def far_frames():
    """A camera 20 m in front of a 16 m volume of 25 cm voxels near (1e5, -1e5, 1e5), where binary32 resolves 8 mm."""
    c = np.array([1e5, -1e5, 1e5])
    poses = []
    for k in range(3):
        p = np.array(synth.orbit_poses(3, 20.0, 20.0, 25.0)[k], np.float64)
        p[:3, 3] += c
        poses.append(p)
    rng = np.random.default_rng(4)
    return [float(v) for v in np.float32(c - 8.0)], poses, [rng.integers(14000, 26000, (60, 80)).astype(np.uint16) for _ in range(3)]


def inside_a_buffer(d):
    """The image in the middle of a device buffer of other depths."""
    n = d.size
    buf = torch.full((3 * n + 16,), 20000, dtype=torch.int16, device="cuda")
    at = (n + 7) // 8 * 8
    buf[at:at + n] = dev(d).reshape(-1)
    return buf[at:at + n].view(d.shape)


@pytest.mark.parametrize("dims", DIMS)
def test_volume_far_from_the_origin(dims):
    """Where a brick's projected corners no longer bound its voxels' pixels:
    every voxel is tested (footprint_bound.h), in this volume and in a handle's."""
    s = 0.25
    org, poses, frames = far_frames()
    o = oracle.Oracle(dims, dims, s, 3 * s, 10, n_threads=8, origin=org)
    F, W = (torch.from_numpy(a).cuda() for a in zeros(dims))
    rgb, Tdr = np.zeros((120, 160, 3), np.uint8), synth.rig_depth_to_rgb()
    Kr = synth.intrinsics(120.0, 110.0, 79.0, 59.0)
    forms = [dict(culling=True), dict(culling=False), dict(schedule=T.TSDF_SCHEDULE_FUSED)]
    vols = [T.Volume(dims, dims, s, 3 * s, 10, origin=org, **f) for f in forms]
    n = 0
    for d, pose in zip(frames, poses):
        dd = inside_a_buffer(d)
        T.tsdf_integrate_geometry_static(dims, s, 3 * s, 10, org, F, W, dd, K, pose)
        torch.cuda.synchronize()
        for v in vols:
            v.integrate(dd, rgb, K, Kr, pose, Tdr)
            v.synchronize()
        n += o.integrate_geometry(d, K, pose)
    assert n > o.F.size // 10
    np.testing.assert_array_equal(W.cpu().numpy(), o.W)
    np.testing.assert_array_equal(F.cpu().numpy(), o.F)
    for v in vols:
        got = v.read()
        v.close()
        np.testing.assert_array_equal(got[1], o.W)
        np.testing.assert_array_equal(got[0], o.F)


@pytest.mark.parametrize("dims", DIMS)
def test_coordinates_that_overflow(dims):
    """Voxel centres at infinity have no camera depth: nothing is updated."""
    F0, W0 = zeros(dims)
    F0 += 0.5
    W0 += 3
    pose = np.eye(4, dtype=np.float32)
    assert check(dims, 1e37, F0, W0, [inside_a_buffer(surface(0)).cpu().numpy().view(np.uint16)], K, [pose],
                 origin=[3e38, 3e38, 3e38]) == 0


SKEWED = {"skew": [[60.0, 3.0, 39.0], [1.5, 55.0, 29.0], [0.0, 0.0, 1.0]],
          "tilted": [[60.0, 0.5, 39.0], [0.2, 55.0, 29.0], [0.05, -0.03, 1.1]]}


@pytest.mark.parametrize("form", sorted(SKEWED))
@pytest.mark.parametrize("dims", DIMS)
def test_depth_camera_that_is_no_pinhole(dims, form):
    s = float(np.float32(0.6 / max(dims)))
    Kd = np.array(SKEWED[form], np.float32)
    F0, W0 = zeros(dims)
    assert check(dims, s, F0, W0, [surface(k) for k in range(3)], Kd, POSES) > F0.size // 20


@pytest.mark.parametrize("dims", [(256, 256, 256), (256, 256, 264), (253, 250, 264)])
def test_culling_on_both_sides_of_the_eight_lane_form(dims):
    """32,768 bricks (the last of the eight-lane form) and 33,792, in whole bricks and ragged ones."""
    s = float(np.float32(1.0 / 264))
    seq = synth.sequence_small(n_frames=2, seed=11)
    F0, W0 = zeros(dims)
    frames = [seq.frame(k)[0] for k in range(2)]
    assert check(dims, s, F0, W0, frames, seq.K_depth, seq.poses) > 10000
    outs = []
    for culling in (True, False):
        with T.Volume(dims, dims, s, 3 * s, 64, culling=culling) as v:
            for k in range(2):
                v.integrate(*seq.frame(k), seq.K_depth, seq.K_rgb, seq.poses[k], seq.T_depth_rgb)
            outs.append(v.read())
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)


def test_captured_calls():
    """Two chained calls captured in a graph, replayed on other depths."""
    dims, s = (64, 64, 64), float(np.float32(0.6 / 64))
    org = [-0.5 * m * s for m in dims]
    F, W = (torch.from_numpy(a).cuda() for a in zeros(dims))
    d = [dev(surface(k)) for k in range(2)]
    call = lambda k, st: T.tsdf_integrate_geometry_static(dims, s, 3 * s, 64, org, F, W, d[k], K, POSES[k], st)  # noqa: E731
    call(0, torch.cuda.current_stream().cuda_stream)  # the scratch array's address is looked up before a capture
    torch.cuda.synchronize()
    F.zero_(), W.zero_()
    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=st):
        call(0, st.cuda_stream)
        call(1, st.cuda_stream)
    o = oracle.Oracle(dims, dims, s, 3 * s, 64, n_threads=4)
    for r in range(3):
        for k in range(2):
            m = surface(10 * r + k)
            d[k].copy_(dev(m))
            o.integrate_geometry(m, K, POSES[k])
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(W.cpu().numpy(), o.W)
        np.testing.assert_array_equal(F.cpu().numpy(), o.F)


@pytest.mark.parametrize("form", sorted(SKEWED))
@pytest.mark.parametrize("dims", [(32, 32, 32), (30, 21, 43)])
@pytest.mark.parametrize("mm", [0, 2500])
def test_handle_with_a_depth_camera_that_is_no_pinhole(dims, form, mm):
    """mm 2500: a wall behind the volume, so its bricks lie in front of every measurement."""
    s = float(np.float32(0.6 / max(dims)))
    Kd = np.array(SKEWED[form], np.float32)
    Kr, Tdr = synth.intrinsics(120.0, 110.0, 79.0, 59.0), synth.rig_depth_to_rgb()
    rgb = np.random.default_rng(5).integers(0, 256, (120, 160, 3)).astype(np.uint8)
    frames = []
    for k in range(6):
        d = surface(k)
        frames.append(np.where(d > 0, mm, 0).astype(np.uint16) if mm else d)
    o = oracle.Oracle(dims, dims, s, 3 * s, 4, n_threads=4)
    for k, d in enumerate(frames):
        o.integrate(d, rgb, Kd, Kr, POSES[k % 3], Tdr)
    assert (o.W > 0).mean() > 0.2
    for form in ("chain", "dense", "batch"):
        with T.Volume(dims, dims, s, 3 * s, 4, culling=form != "dense") as v:
            b = T.Batch([v]) if form == "batch" else None
            for k, d in enumerate(frames):
                if b:
                    b.integrate([(dev(d), torch.from_numpy(rgb).cuda(), Kd, Kr, POSES[k % 3], Tdr)])
                    b.synchronize()
                else:
                    v.integrate(d, rgb, Kd, Kr, POSES[k % 3], Tdr)
            got = v.read()
            if b:
                b.close()
        np.testing.assert_array_equal(got[1], o.W, err_msg=form)
        np.testing.assert_array_equal(got[0], o.F, err_msg=form)
        np.testing.assert_array_equal(got[2], o.C, err_msg=form)
