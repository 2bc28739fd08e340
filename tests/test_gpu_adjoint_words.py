"""The adjoint's two access widths: images that start on a 16-byte boundary and
hold whole 16-byte words, and others, give the same colours and camera
gradients bit for bit and the same image gradient to the order of its
additions; the camera sums equal those of a binary64 evaluation."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1602_06645_gb300 as T  # noqa: E402
from paper_1602_06645_gb300 import synth  # noqa: E402
from paper_1602_06645_gb300.adjoint import Adjoint  # noqa: E402


@pytest.mark.parametrize("w,h,n", [(320, 180, 4), (321, 179, 3)])  # 321 x 179 x 3 x 3 floats are no whole words
def test_access_widths_agree(w, h, n):
    seq = synth.sequence_adjoint(n_frames=n, dims_geo=48)
    K4 = np.array([1050.0 * w / 1920, 1050.0 * w / 1920, (w - 1) / 2, (h - 1) / 2], np.float32)
    Tm = np.asarray(seq.T_depth_rgb, np.float32)
    with T.Volume(seq.dims_geo, seq.dims_col, seq.voxel_size, seq.mu, seq.max_weight) as vol:
        adj = Adjoint(vol, n, max_pairs=1 << 20)
        for f in range(n):
            adj.record(seq.frame(f)[0], seq.K_depth, seq.poses[f])
        nv = adj.finalize()
        assert nv > 1000
        rng = np.random.default_rng(w)
        images = rng.uniform(0, 255, (n, h, w, 3)).astype(np.float32)
        g = torch.from_numpy(rng.normal(size=(nv, 3)).astype(np.float32)).cuda()
        got = []
        for shift in (0, 1, 2, 3):  # floats after a 16-byte boundary
            def placed(a):
                buf = torch.zeros(a.size + 8, device="cuda")
                t = buf[shift:shift + a.size].view(a.shape)
                t.copy_(torch.from_numpy(a))
                return buf, t
            ibuf, im = placed(images)
            gbuf, gi = placed(np.zeros_like(images))
            C, cnt = adj.forward(im, K4, Tm)
            theta = adj.backward(im, K4, Tm, g, gi)
            got.append((C.cpu().numpy(), cnt.cpu().numpy(), theta, gi.cpu().numpy()))
            # nothing outside the image gradient is written
            assert not gbuf[:shift].any() and not gbuf[shift + images.size:].any()
        for C, cnt, theta, gi in got[1:]:
            np.testing.assert_array_equal(C, got[0][0])
            np.testing.assert_array_equal(cnt, got[0][1])
            np.testing.assert_array_equal(theta, got[0][2])
            # a pixel's few dozen additions in another order: each rounds by 2^-24 of the partial sum
            np.testing.assert_allclose(gi, got[0][3], rtol=0, atol=64 * 2.0 ** -24 * np.abs(got[0][3]).max())
        # every gradient of a voxel reaches the images once: the weights of a footprint add up to 1
        has = got[0][1] > 0
        want = g.cpu().numpy().astype(np.float64)[has].sum(0)
        have = got[0][3].astype(np.float64).sum((0, 1, 2))
        scale = np.abs(g.cpu().numpy()[has]).sum()
        np.testing.assert_allclose(have, want, rtol=0, atol=16 * 2.0 ** -24 * scale)
        adj.close()
