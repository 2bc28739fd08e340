"""A restore that fails half way (no memory for a staging buffer) has changed F
but not w: what the handle remembers of the bricks must be that of the values
it now holds, so that later frames give what the dense sweep gives."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1602_06645_gb300 as T  # noqa: E402
from paper_1602_06645_gb300 import synth  # noqa: E402


class Failing:
    """PyTorch's allocator, which refuses the n-th allocation from `arm` on."""

    def __init__(self):
        self.inner = T.torch_allocator()
        self.left = None

        def alloc(nbytes, stream, ctx):
            if self.left is not None:
                self.left -= 1
                if self.left < 0:
                    return None
            return self.inner.alloc(nbytes, stream, ctx)

        def free(ptr, nbytes, stream, ctx):
            self.inner.free(ptr, nbytes, stream, ctx)

        self.c = T.tsdf_allocator(T.ALLOC_FN(alloc), T.FREE_FN(free), None)


@pytest.mark.parametrize("bad", ["half", "nan"])
def test_frames_after_a_failed_restore_equal_the_dense_sweep(bad):
    dims, s = (32, 32, 32), float(np.float32(0.6 / 32))
    K, Kr, Tdr = synth.intrinsics(60.0, 55.0, 39.0, 29.0), synth.intrinsics(120.0, 110.0, 79.0, 59.0), synth.rig_depth_to_rgb()
    poses = synth.orbit_poses(3, 0.9, 20.0, 25.0)
    rgb = np.zeros((120, 160, 3), np.uint8)
    wall = np.full((60, 80), 2500, np.uint16)
    rng = np.random.default_rng(3)
    F0 = rng.uniform(-0.5, 0.5, dims).astype(np.float32)
    if bad == "nan":
        F0.reshape(-1)[::37] = np.nan
    outs = []
    for culling in (1, 0):
        a = Failing()
        p = T.tsdf_params_default()
        p.culling, p.allocator = culling, a.c
        p.stream = torch.cuda.current_stream().cuda_stream
        h = T.tsdf_create_ex(dims, dims, s, 3 * s, 64, p)
        try:
            for k in range(3):
                T.tsdf_integrate(h, wall, rgb, K, Kr, poses[k], Tdr)
            W0 = np.empty(dims, np.uint8)
            T.tsdf_read(h, None, W0)
            a.left = 1  # F's staging buffer is there, w's is not
            with pytest.raises(T.TsdfError) as e:
                T.tsdf_write(h, F0, np.zeros(dims, np.uint8))
            assert e.value.status == T.TSDF_ERR_OOM
            a.left = None
            T.tsdf_synchronize(h)
            views = []
            with T.Volume(dims, dims, s, 3 * s, 64) as same:  # the same values, restored without a failure
                same.write(F0, W0)
                for g in (h, same.h):
                    r, vx, nm = (np.empty((60, 80) + c, np.float32) for c in ((), (3,), (3,)))
                    T.tsdf_raycast(g, K, poses[0], (80, 60), range_=r, vertex=vx, normal=nm)
                    views.append((r, vx, nm))
            for x, y in zip(*views):
                np.testing.assert_array_equal(x, y)
            for k in range(3):
                T.tsdf_integrate(h, wall, rgb, K, Kr, poses[k], Tdr)
            F, W = np.empty(dims, np.float32), np.empty(dims, np.uint8)
            T.tsdf_read(h, F, W)
            outs.append((F, W))
        finally:
            T.tsdf_destroy(h)
    for x, y in zip(*outs):
        np.testing.assert_array_equal(x, y)
