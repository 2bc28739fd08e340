"""Read-out and restore of the volumes between linear arrays and the library's
layout, at the access widths that row length and address allow, and the brick
summaries that a restore recomputes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1602_06645_gb300 as T  # noqa: E402
from paper_1602_06645_gb300 import synth  # noqa: E402


def shifted(a, by):
    """The array on the device, `by` elements after a 256-byte boundary."""
    t = torch.from_numpy(a)
    buf = torch.empty(a.size + by, dtype=t.dtype, device="cuda")
    out = buf[by:].view(a.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("shift", [0, 1, 2, 4])
@pytest.mark.parametrize("nx", [1, 2, 7, 8, 12, 31, 32, 33, 64, 66, 130])
def test_restore_and_read_are_exact(nx, shift):
    g, c = (nx, 9, 17), (2 * nx, 18, 34)
    rng = np.random.default_rng(nx * 8 + shift)
    F = rng.uniform(-1, 1, g[::-1]).astype(np.float32)
    W = rng.integers(0, 256, g[::-1]).astype(np.uint8)
    C = rng.integers(0, 1 << 31, c[::-1]).astype(np.int32)
    with T.Volume(g, c, 0.01, 0.03, 64) as v:
        v.write(shifted(F, shift), shifted(W, shift), shifted(C, shift))
        for got, want in zip(v.read(), (F, W, C.view(np.uint32))):  # host arrays, slab by slab
            np.testing.assert_array_equal(got, want)
        out = [shifted(np.zeros_like(a), shift) for a in (F, W, C)]
        T.tsdf_read(v.h, *out)
        for got, want in zip(out, (F, W, C)):
            np.testing.assert_array_equal(got.cpu().numpy(), want)
        v.write(F[::-1].copy(), W[::-1].copy(), C[::-1].copy())  # from host arrays
        for got, want in zip(v.read_torch(), (F[::-1], W[::-1], C[::-1])):
            np.testing.assert_array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("n", [24, 29])
def test_restored_summaries_lose_no_brick(n):
    """Frames fused after a restore, with the culling that reads the summaries
    and without: the same volumes (observed and unobserved voxels, bricks
    on one side of the band, saturated free space)."""
    rng = np.random.default_rng(n)
    F = np.ones((n, n, n), np.float32)
    F[: n // 2] = rng.uniform(-1, 1, (n // 2, n, n)).astype(np.float32)
    W = rng.integers(0, 3, (n, n, n)).astype(np.uint8) * 32
    W[:, :, : n // 3] = 64
    seq = synth.sequence_small(n_frames=2, dims_geo=24, seed=3)
    frames = [seq.frame(f) for f in range(2)]
    outs = []
    for culling in (True, False):
        with T.Volume((n,) * 3, (2 * n,) * 3, 1.0 / n, 3.0 / n, 64, culling=culling) as v:
            v.write(F, W)
            for f, (d, c) in enumerate(frames):
                v.integrate(d, c, seq.K_depth, seq.K_rgb, seq.poses[f], seq.T_depth_rgb)
            outs.append(v.read())
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)
    assert ((outs[0][2] >> 24) > 0).sum() > 100
