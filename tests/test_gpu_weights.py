"""Weights above the weight limit, which a caller may hand over (an array of
another program, a limit lowered between calls, tsdf_write, tsdf_load): the
update takes them to min(w + 1, max_weight) and leaves every other voxel's
weight alone, in caller-owned volumes of any alignment and in handles by every
schedule, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1602_06645_gb300 as T  # noqa: E402
from paper_1602_06645_gb300 import synth  # noqa: E402

K, KR = synth.intrinsics(60.0, 55.0, 39.0, 29.0), synth.intrinsics(120.0, 110.0, 79.0, 59.0)
TDR = synth.rig_depth_to_rgb()
POSES = synth.orbit_poses(3, 0.9, 20.0, 25.0)


def volume(dims, seed, ones=False):
    """F and w with every weight 0..255 among them, an unobserved voxel in every brick."""
    rng = np.random.default_rng(seed)
    shape = dims[::-1]
    W = rng.integers(0, 256, shape).astype(np.uint8)
    W[::5, ::5, ::5] = 0
    F = np.ones(shape, np.float32) if ones else rng.uniform(-1, 1, shape).astype(np.float32)
    return F, W


def depth(mm, seed):
    """A wall of mm millimetres (0: one that cuts the volume) with some gaps."""
    rng = np.random.default_rng(seed)
    d = np.full((60, 80), mm, np.uint16) if mm else rng.integers(700, 1100, (60, 80)).astype(np.uint16)
    d[rng.random((60, 80)) < 0.05] = 0
    return d


@pytest.mark.parametrize("max_weight", [1, 64, 128, 255])
@pytest.mark.parametrize("dims", [(64, 64, 64), (36, 29, 43), (37, 30, 41)])
@pytest.mark.parametrize("shift", [0, 1])
def test_caller_owned_weights_above_the_limit(dims, shift, max_weight):
    s = float(np.float32(0.6 / max(dims)))
    n = dims[0] * dims[1] * dims[2]
    F0, W0 = volume(dims, max_weight)
    F = torch.zeros(n + 16, device="cuda")[shift:shift + n]
    W = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")[shift:shift + n]
    F.copy_(torch.from_numpy(F0.reshape(-1))), W.copy_(torch.from_numpy(W0.reshape(-1)))
    o = oracle.Oracle(dims, dims, s, 3 * s, max_weight, n_threads=4)
    o.F[...], o.W[...] = F0, W0
    for k in range(3):
        d = depth(0, k)
        T.tsdf_integrate_geometry_static(dims, s, 3 * s, max_weight, [-0.5 * m * s for m in dims], F, W,
                                         torch.from_numpy(d.view(np.int16)).cuda(), K, POSES[k])
        assert o.integrate_geometry(d, K, POSES[k]) > n // 20
    torch.cuda.synchronize()
    np.testing.assert_array_equal(W.cpu().numpy().reshape(o.W.shape), o.W)
    np.testing.assert_array_equal(F.cpu().numpy().reshape(o.F.shape), o.F)


@pytest.mark.parametrize("max_weight", [1, 64, 128, 255])
@pytest.mark.parametrize("dims", [(32, 32, 32), (30, 21, 43)])
@pytest.mark.parametrize("mode", ["surface", "open", "no_free_space"])
def test_handle_weights_above_the_limit(dims, mode, max_weight):
    s = float(np.float32(0.6 / max(dims)))
    F0, W0 = volume(dims, max_weight, ones=mode == "open")  # open: F = 1 in front of every measurement
    rgb = np.zeros((120, 160, 3), np.uint8)
    free = mode != "no_free_space"
    frames = [depth(2500 if mode == "open" else 0, k) for k in range(3)]
    o = oracle.Oracle(dims, dims, s, 3 * s, max_weight, n_threads=4, update_free_space=int(free))
    o.F[...], o.W[...] = F0, W0
    for k, d in enumerate(frames):
        o.integrate(d, rgb, K, KR, POSES[k], TDR)
    kw = dict(update_free_space=free)
    for form in (dict(culling=True), dict(culling=False), dict(schedule=T.TSDF_SCHEDULE_FUSED), "batch"):
        with T.Volume(dims, dims, s, 3 * s, max_weight, **kw, **({} if form == "batch" else form)) as v:
            v.write(F0, W0)
            if form == "batch":
                b = T.Batch([v])
                for k, d in enumerate(frames):
                    b.integrate([(torch.from_numpy(d.view(np.int16)).cuda(), torch.from_numpy(rgb).cuda(), K, KR,
                                  POSES[k], TDR)])
                    b.synchronize()
                b.close()
            else:
                for k, d in enumerate(frames):
                    v.integrate(d, rgb, K, KR, POSES[k], TDR)
            F, W, _ = v.read()
        np.testing.assert_array_equal(W, o.W, err_msg=str(form))
        np.testing.assert_array_equal(F, o.F, err_msg=str(form))


@pytest.mark.parametrize("above", [0, 3, 191])
@pytest.mark.parametrize("dims", [(32, 32, 32), (30, 21, 43)])
def test_free_space_above_the_limit_is_not_saturated(dims, above):
    """Free space (F = 1) whose smallest weight is the limit: it is left out of
    the update only where no weight lies above the limit."""
    s, limit = float(np.float32(0.6 / max(dims))), 64
    shape = dims[::-1]
    F0, W0 = np.ones(shape, np.float32), np.full(shape, limit, np.uint8)
    W0[::5, ::3, ::5] += above
    rgb = np.zeros((120, 160, 3), np.uint8)
    o = oracle.Oracle(dims, dims, s, 3 * s, limit, n_threads=4)
    o.F[...], o.W[...] = F0, W0
    for k in range(2):
        o.integrate(depth(2500, k), rgb, K, KR, POSES[k], TDR)
    assert above == 0 or ((o.W == limit) & (W0 > limit)).sum() > 100
    for form in (dict(culling=True), dict(culling=False), dict(schedule=T.TSDF_SCHEDULE_FUSED)):
        with T.Volume(dims, dims, s, 3 * s, limit, **form) as v:
            v.write(F0, W0)
            for k in range(2):
                v.integrate(depth(2500, k), rgb, K, KR, POSES[k], TDR)
            F, W, _ = v.read()
            if form.get("culling") and above == 0:
                assert v.stats().geo_bricks == 0  # saturated free space
        np.testing.assert_array_equal(W, o.W, err_msg=str(form))
        np.testing.assert_array_equal(F, o.F, err_msg=str(form))
