"""Ray casting across uniform space (free and unobserved cubes of bricks that
the march crosses without sampling) against the oracle, which samples every
step: bit for bit."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1602_06645_gb300 as T  # noqa: E402
from paper_1602_06645_gb300 import synth  # noqa: E402


def volume(dims, kind, s):
    """F, W, C (z, y, x): two spheres in wholly observed free space, with the
    inside unobserved beyond the band, and by kind a hole of unobserved voxels
    (a slab of bricks, single voxels) or odd values."""
    x, y, z = (-0.5 * n * s + (np.arange(n) + 0.5) * s for n in dims)
    z, y, x = np.meshgrid(z, y, x, indexing="ij")
    e = s * min(dims)
    sd = np.minimum(np.sqrt((x - 0.1 * e) ** 2 + y ** 2 + z ** 2) - 0.2 * e,
                    np.sqrt((x + 0.25 * e) ** 2 + (y - 0.2 * e) ** 2 + z ** 2) - 0.1 * e)
    F = np.clip(sd / (3 * s), -1.0, 1.0).astype(np.float32)
    W = np.where(sd < -3 * s, 0, 5).astype(np.uint8)
    rng = np.random.default_rng(sum(dims))
    if kind == "slab":
        W[:, : dims[1] // 4] = 0
    if kind == "specks":
        W[rng.random(W.shape) < 0.002] = 0
    if kind == "odd":  # beside free space, in bricks that hold other values too
        at = np.argwhere((sd > 0) & (sd < 3 * s))[::37]
        F[tuple(at.T)] = np.resize(np.array([np.nan, np.inf, -np.inf, 3e38], np.float32), len(at))
    C = rng.integers(0, 1 << 32, W.shape, dtype=np.uint32)
    return F, W, C


CAMERAS = {
    "outside": synth.look_at((0.9, 0.5, 0.6), (0.0, 0.0, 0.0)),
    "inside": synth.look_at((0.3, -0.3, 0.28), (0.0, 0.05, 0.0)),
    "axis": synth.look_at((0.0, 1.2, 0.0), (0.0, 0.0, 0.0)),
    "away": synth.look_at((0.9, 0.5, 0.6), (1.8, 1.0, 1.2)),
}


@pytest.mark.parametrize("dims", [(96, 96, 96), (70, 45, 83), (8, 8, 8), (9, 2, 130)])
@pytest.mark.parametrize("kind", ["whole", "slab", "specks", "odd"])
@pytest.mark.parametrize("camera", list(CAMERAS))
def test_cast_equals_oracle(dims, kind, camera):
    s = float(np.float32(1.0 / max(dims)))
    F, W, C = volume(dims, kind, s)
    K = synth.intrinsics(70.0, 75.0, 39.5, 29.5)
    with T.Volume(dims, dims, s, 3 * s, 64) as vol:
        vol.write(F, W, C)
        info = vol.info()
        for steps in ((1.5, 0.5), (0.3, 0.3), (7.0, 0.5)):
            a = (K, CAMERAS[camera], (83, 61), 0.01, 2.5, float(np.float32(steps[0] * s)), float(np.float32(steps[1] * s)))
            g = vol.raycast(*a)
            o = oracle.raycast(F, W, C, s, s, info.origin, *a)
            for k in ("range", "vertex", "normal", "rgbw"):
                np.testing.assert_array_equal(g[k], o[k], err_msg="%s, steps %s" % (k, steps))


def test_cast_far_from_the_world_origin_equals_oracle():
    """Where a sample's position is rounded to a good part of a voxel."""
    dims, s = (64, 64, 64), float(np.float32(1.0 / 64))
    F, W, C = volume(dims, "whole", s)
    K = synth.intrinsics(70.0, 75.0, 39.5, 29.5)
    for shift in (1e3, 3e4):
        cam = CAMERAS["outside"].copy()
        cam[:3, 3] += np.float32(shift)
        with T.Volume(dims, dims, s, 3 * s, 64, origin=[shift - 0.5] * 3) as vol:
            vol.write(F, W, C)
            a = (K, cam, (83, 61), 0.01, 2.5, float(np.float32(1.5 * s)), float(np.float32(0.5 * s)))
            g = vol.raycast(*a)
            o = oracle.raycast(F, W, C, s, s, vol.info().origin, *a)
            for k in ("range", "vertex", "normal", "rgbw"):
                np.testing.assert_array_equal(g[k], o[k], err_msg="%s at %g" % (k, shift))
            assert o["hits"] > 100
