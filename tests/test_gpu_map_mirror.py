"""The map kernel that evaluates a half or a quarter of the tiles and writes
their mirror images, against the one that evaluates every tile (a map with
derivatives takes that), bit for bit; and its tile cones through a raster on
the same map uploaded, whose cones are reduced from all pixels.  Sizes: whole
tiles in x, in y, in both, in neither; odd and even tile counts, one tile."""
import numpy as np
import pytest

from paper_2003_10558_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(16, 16), (32, 16), (48, 80), (64, 37), (37, 64), (49, 33), (160, 96), (176, 91), (1, 16), (16, 1)]
LENSES = [(0.32, 0.62, 0.86, 270.0, 0), (0.0, 1.0, 1.0, 180.0, 1), (-0.7, 0.8, 0.6, 240.0, 0), (1.0, 0.0, 0.5, 120.0, 2)]


@pytest.fixture(scope="module")
def vsr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_10558_gb300 import build, vsr as V
    build.build()
    V.load()
    return V


@pytest.mark.parametrize("W,H", SIZES)
def test_mirrored_map(vsr, W, H):
    tris = torch.from_numpy(scenes.random_triangles(2000, 1.0, 20.0, 0.1, seed=W + H)).cuda()
    for k, l, s, om, aov in LENSES:
        m = vsr.Map(W, H, k, l, s, om, aov)
        full = vsr.Map.from_spec(vsr.MAP_UNIVERSAL, W, H, (k, l, s, om), aov=aov, derivatives=True)
        a, b = m.download(), full.download()
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32)), (k, aov)
        up = vsr.Map.from_tensor(torch.from_numpy(a).cuda())
        x = vsr.raster(m, vsr.Scene(tris))
        y = vsr.raster(up, vsr.Scene(tris))
        # the tile axes differ in their last bits: rounding of the distances
        # in ramp units, tile size x 2^-23 and a few roundings
        assert (x["cov"] - y["cov"]).abs().max().item() <= 1e-5
        assert (x["id"] != y["id"]).float().mean().item() <= 1e-4 or W * H < 10_000 and (x["id"] != y["id"]).sum() <= 1
    assert vsr.last_device_status() == 0
