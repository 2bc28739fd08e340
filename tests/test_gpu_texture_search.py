"""Texel fill finds each texel's triangle: layouts of the library and layouts of
the caller's with single-texel-row, large and empty maps, against a plain
evaluation of every texel on its own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1602_06645_gb300 as T  # noqa: E402


@pytest.fixture(scope="module")
def volume():
    n = 24
    v = T.Volume((n,) * 3, (n,) * 3, 1.0 / n, 3.0 / n, 64)
    rng = np.random.default_rng(4)
    C = rng.integers(0, 1 << 24, (n,) * 3, dtype=np.uint32) | np.where(rng.random((n,) * 3) < 0.9, 7 << 24, 0).astype(np.uint32)
    v.write(None, None, C)
    yield v
    v.close()


@pytest.mark.parametrize("n,kind", [(1, "plain"), (33, "plain"), (2000, "plain"), (700, "empty runs"), (1500, "mixed"),
                                    (40, "large")])
def test_every_texel_reads_its_own_triangle(volume, n, kind):
    rng = np.random.default_rng(n)
    tris = rng.uniform(-0.45, 0.45, (n, 9)).astype(np.float32)
    lo, hi = (40, 90) if kind == "large" else (2, 5)
    wh = rng.integers(lo, hi, (n, 2)).astype(np.int32)
    if kind == "mixed":
        wh[rng.random(n) < 0.05] = (61, 37)
    sizes = wh.prod(1).astype(np.int64)
    if kind == "empty runs":  # offsets that give long runs of triangles no texel
        sizes[100:400] = 0
        sizes[rng.random(n) < 0.3] = 0
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    total = int(off[-1])
    tex = torch.full((total + 64,), -1, dtype=torch.int32, device="cuda")
    dev = [torch.from_numpy(a).cuda() for a in (tris, wh, off)]
    T.tsdf_texture_fill(volume.h, dev[0], n, dev[1], dev[2], tex)
    got = tex.cpu().numpy()
    assert (got[total:] == -1).all()
    # each triangle alone: the same texels, with no search to do
    for t in list(range(0, n, max(1, n // 60))) + [n - 1]:
        if sizes[t] == 0:
            continue
        one = np.empty(sizes[t], np.uint32)
        T.tsdf_texture_fill(volume.h, tris[t:t + 1], 1, wh[t:t + 1], np.array([0, sizes[t]], np.int64), one)
        np.testing.assert_array_equal(got[off[t]:off[t + 1]].view(np.uint32), one)
