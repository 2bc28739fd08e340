"""Bricks in front of every measurement, whose update only counts weights,
against the general update (the dense sweep takes it for every brick) and the
oracle: first observations, gaps in the depth image, weights up to the limit,
ragged volumes, restored values that the shorter update must leave alone."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1602_06645_gb300 as T  # noqa: E402
from paper_1602_06645_gb300 import synth  # noqa: E402


def wall(shape, mm, gaps, seed):
    """A wall at mm millimetres with a share of pixels without depth."""
    rng = np.random.default_rng(seed)
    d = np.full(shape, mm, np.uint16)
    d[rng.random(shape) < gaps] = 0
    return d


@pytest.mark.parametrize("dims", [(32, 32, 32), (30, 21, 43), (1, 9, 64)])
@pytest.mark.parametrize("gaps", [0.0, 0.02, 0.6])
@pytest.mark.parametrize("restored", ["empty", "ones", "mixed", "odd"])
def test_open_bricks_equal_general_update(dims, gaps, restored):
    s = float(np.float32(0.6 / max(dims)))
    shape = dims[::-1]
    rng = np.random.default_rng(sum(dims))
    F, W = np.zeros(shape, np.float32), np.zeros(shape, np.uint8)
    if restored != "empty":
        W = rng.integers(0, 9, shape).astype(np.uint8)
        F = np.where(W > 0, 1.0, 0.25).astype(np.float32)  # an unobserved voxel keeps what was written
    if restored == "mixed":
        F[:, :, : dims[0] // 2] = rng.uniform(-1, 1, F[:, :, : dims[0] // 2].shape)
    if restored == "odd":  # the shorter update takes none of these volumes
        F.reshape(-1)[:: 61] = np.resize(np.array([np.nan, np.inf, 3e38], np.float32), F.reshape(-1)[:: 61].shape)
    K = synth.intrinsics(60.0, 55.0, 39.0, 29.0)
    Kr, Tdr = synth.intrinsics(120.0, 110.0, 79.0, 59.0), synth.rig_depth_to_rgb()
    poses = synth.orbit_poses(3, 0.9, 20.0, 25.0)
    rgb = rng.integers(0, 256, (120, 160, 3)).astype(np.uint8)
    outs = []
    for culling in (True, False):
        with T.Volume(dims, dims, s, 3 * s, 10, culling=culling) as v:
            v.write(F, W)
            for k in range(12):  # past the weight limit
                v.integrate(wall((60, 80), 2500, gaps, k), rgb, K, Kr, poses[k % 3], Tdr)
            outs.append(v.read())
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)
    if restored == "empty":
        o = oracle.Oracle(dims, dims, s, 3 * s, 10, n_threads=4)
        for k in range(12):
            o.integrate(wall((60, 80), 2500, gaps, k), rgb, K, Kr, poses[k % 3], Tdr)
        np.testing.assert_array_equal(outs[0][0], o.F)
        np.testing.assert_array_equal(outs[0][1], o.W)
        assert (o.W > 0).mean() > 0.3


def test_open_bricks_in_a_batch_equal_the_frame_by_frame_update():
    dims, s = (40, 24, 33), float(np.float32(0.6 / 40))
    K, Kr, Tdr = synth.intrinsics(60.0, 55.0, 39.0, 29.0), synth.intrinsics(120.0, 110.0, 79.0, 59.0), synth.rig_depth_to_rgb()
    poses = synth.orbit_poses(3, 0.9, 20.0, 25.0)
    rgb = torch.zeros((120, 160, 3), dtype=torch.uint8, device="cuda")
    vols = [T.Volume(d, d, s, 3 * s, 10) for d in (dims, (32, 32, 32))]
    alone = [T.Volume(d, d, s, 3 * s, 10) for d in (dims, (32, 32, 32))]
    b = T.Batch(vols)
    for k in range(4):
        depth = torch.from_numpy(wall((60, 80), 2500, 0.02, k).view(np.int16)).cuda()
        torch.cuda.synchronize()
        b.integrate([(depth, rgb, K, Kr, poses[k % 3], Tdr)] * 2)
        for v in alone:
            v.integrate(depth, rgb, K, Kr, poses[k % 3], Tdr)
    b.synchronize()
    for v, a in zip(vols, alone):
        for x, y in zip(v.read(), a.read()):
            np.testing.assert_array_equal(x, y)
        assert v.stats().total_geo_bricks == a.stats().total_geo_bricks > 0
        assert v.stats().total_geo_updated == a.stats().total_geo_updated
    b.close()
