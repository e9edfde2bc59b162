"""Workspace that is allocated while a stream captures (relaxed mode, which
allows it) serves eager frames before the graph's first launch, and the
graph's launches after them."""
import numpy as np
import pytest

from paper_2003_10558_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vsr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_10558_gb300 import build, vsr as V
    build.build()
    V.load()
    return V


def _crowd(n, spread, seed):
    """n small triangles around world +z: tiles shared between CTAs."""
    t = scenes.random_triangles(n, 2.0, 20.0, 0.01, seed).astype(np.float64)
    c = t.mean(axis=1, keepdims=True)
    rng = np.random.default_rng(seed)
    d = np.stack([rng.normal(0, spread, n), rng.normal(0, spread, n), np.ones(n)], 1)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return (t - c + np.linalg.norm(c, axis=2, keepdims=True) * d[:, None, :]).astype(np.float32)


@pytest.mark.parametrize("what", ["set-up", "walk", "items"])
def test_eager_frames_before_the_first_launch(vsr, what):
    tris = torch.from_numpy(_crowd(12_000, 0.05, 10)).cuda()
    m = vsr.Map(96, 80, 0.0, 1.0, 1.0, 40.0)
    ref = vsr.raster_dense(m, vsr.Scene(tris, scenes.camera()))
    out = {key: torch.zeros_like(t) for key, t in ref.items()}
    sc = vsr.Scene()
    if what != "set-up":  # known shape, but nothing rasterized
        sc.update(tris, scenes.camera())
        vsr.bin(m, sc)

    def frame(o):
        if what == "set-up":
            sc.update(tris, scenes.camera())
        elif what == "walk":
            vsr.raster(m, sc, out=o)
        else:
            vsr.raster(m, sc, out=o, binned=True)

    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        frame(out)
    for q in range(3):
        o = {key: torch.zeros_like(t) for key, t in ref.items()}
        frame(o)
        if what == "set-up":
            vsr.raster(m, sc, out=o)
        for key in ref:
            assert torch.equal(o[key].view(torch.int32), ref[key].view(torch.int32)), (q, key)
        g.replay()
        if what == "set-up":
            vsr.raster(m, sc, out=out)
        torch.cuda.synchronize()
        for key in ref:
            assert torch.equal(out[key].view(torch.int32), ref[key].view(torch.int32)), (q, key)
    assert vsr.last_device_status() == 0
