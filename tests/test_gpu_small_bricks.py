"""Brick culling by eight lanes per brick (small volumes) and by one thread
(larger ones), and the caller-owned volume's two access widths, against the
oracle and the dense sweep."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1602_06645_gb300 as T  # noqa: E402
from paper_1602_06645_gb300 import synth  # noqa: E402


def frames(seed, n=3):
    seq = synth.sequence_small(n_frames=n, seed=seed)
    return seq, [seq.frame(f) for f in range(n)]


# 65,536 bricks is the largest volume of the eight-lane form
@pytest.mark.parametrize("dims", [(8, 8, 8), (40, 33, 57), (512, 512, 128), (512, 512, 136), (1000, 16, 24)])
@pytest.mark.parametrize("view", ["orbit", "inside", "away"])
def test_culling_equals_dense_sweep(dims, view):
    seq, fr = frames(7)
    s = float(np.float32(1.0 / max(dims)))
    poses = {"orbit": seq.poses, "inside": [synth.look_at((0.05, 0.02, 0.04), (0.3, 0.1, -0.2))] * 3,
             "away": [synth.look_at((0.6, 0.0, 0.1), (1.4, 0.3, 0.2))] * 3}[view]
    outs = []
    for culling in (True, False):
        with T.Volume(dims, dims, s, 3 * s, 64, culling=culling) as v:
            for k, (d, c) in enumerate(fr):
                v.integrate(d, c, seq.K_depth, seq.K_rgb, poses[k], seq.T_depth_rgb)
            outs.append(v.read())
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("dims", [(64, 64, 64), (36, 29, 43), (37, 30, 41), (4, 3, 2)])
@pytest.mark.parametrize("shift", [0, 1, 4])
def test_caller_owned_volume_at_any_alignment(dims, shift):
    """Rows of a multiple of four voxels on 16-byte boundaries take wide
    accesses, others single voxels: the oracle's volume either way, and nothing
    written around it."""
    seq, fr = frames(9)
    s = float(np.float32(1.0 / max(dims)))
    n = dims[0] * dims[1] * dims[2]
    Fb = torch.full((n + 16,), -7.0, device="cuda")
    Wb = torch.full((n + 16,), 77, dtype=torch.uint8, device="cuda")
    F, W = Fb[shift:shift + n], Wb[shift:shift + n]
    F.zero_(), W.zero_()
    o = oracle.Oracle(dims, dims, s, 3 * s, 2, n_threads=4)
    for k, (d, c) in enumerate(fr):
        T.tsdf_integrate_geometry_static(dims, s, 3 * s, 2, [-0.5 * m * s for m in dims], F, W,
                                         torch.from_numpy(d.view(np.int16)).cuda(), seq.K_depth, seq.poses[k])
        o.integrate(d, c, seq.K_depth, seq.K_rgb, seq.poses[k], seq.T_depth_rgb)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(W.cpu().numpy().reshape(o.W.shape), o.W)
    np.testing.assert_array_equal(F.cpu().numpy().reshape(o.F.shape), o.F)
    assert (Fb[:shift] == -7).all() and (Fb[shift + n:] == -7).all()
    assert (Wb[:shift] == 77).all() and (Wb[shift + n:] == 77).all()
