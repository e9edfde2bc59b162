"""A crowded object in a large picture: tiles of one block of candidates and
more, at the edges of the blocks by which the walking raster shares a tile, and
of more crowded tiles than it has slots.  Every picture is the dense reference
(every pixel x every triangle) bit for bit."""
import numpy as np
import pytest

from paper_2003_10558_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KEYS = ("id", "depth", "cov")


@pytest.fixture(scope="module")
def vsr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_10558_gb300 import build, vsr as V
    build.build()
    V.load()
    return V


def _object(n, spread, jitter, seed):
    """n small triangles in directions around the world's +z axis."""
    t = scenes.random_triangles(n, 2.0, 20.0, jitter, seed).astype(np.float64)
    c = t.mean(axis=1, keepdims=True)
    rng = np.random.default_rng(seed)
    d = np.stack([rng.normal(0, spread, n), rng.normal(0, spread, n), np.ones(n)], 1)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return torch.from_numpy((t - c + np.linalg.norm(c, axis=2, keepdims=True) * d[:, None, :]).astype(np.float32)).cuda()


# 1280 tiles and more are a large picture (160 SMs x 8 CTAs at most)
CASES = [(n, 0.001, 0.01) for n in (1000, 1024, 1025, 1279, 1281, 2048, 2049, 3073)] + [
    (12_000, 0.03, 0.02), (20_000, 0.5, 0.3)]


@pytest.mark.parametrize("n,spread,jitter", CASES)
def test_crowded_tiles_of_a_large_picture(vsr, n, spread, jitter):
    tris = _object(n, spread, jitter, n)
    for W, H in ((720, 512), (1003, 517)):
        m = vsr.Map(W, H, 0.2, 0.9, 0.9, 100.0)
        sc = vsr.Scene(tris, scenes.camera())
        ref = vsr.raster_dense(m, sc)
        for _ in range(3):  # the first frame goes through stored bins
            out = vsr.raster(m, sc)
            for key in KEYS:
                assert torch.equal(out[key].view(torch.int32), ref[key].view(torch.int32)), (W, key)
        pairs = sc.bin_pairs()
        vsr.bin(m, sc)
        assert sc.bin_pairs() == pairs
    assert vsr.last_device_status() == 0
