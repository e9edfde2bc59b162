"""Stored bins and pair counts after frames that stored none: a view that goes
from almost no triangles to most of the scene over frames that bin as they
rasterize, then every call that reads stored bins."""
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


def _half(n, seed):
    """n triangles of which all but a few lie around the world's +z axis."""
    t = scenes.random_triangles(n, 2.0, 20.0, 0.05, seed).astype(np.float64)
    c = t.mean(axis=1, keepdims=True)
    rng = np.random.default_rng(seed)
    d = np.stack([rng.normal(0, 0.2, n), rng.normal(0, 0.2, n), np.ones(n)], 1)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    moved = (t - c + np.linalg.norm(c, axis=2, keepdims=True) * d[:, None, :]).astype(np.float32)
    moved[:50] = scenes.random_triangles(50, 2.0, 20.0, 0.05, seed + 1)
    return moved


def _turned(a):
    """A camera that looks at angle a from +z."""
    c, s = np.cos(a), np.sin(a)
    return scenes.camera((0.0, 0.0, 0.0), np.array([[c, 0.0, s], [0.0, 1.0, 0.0], [-s, 0.0, c]]))


def _equal(a, b):
    for key in KEYS:
        assert torch.equal(a[key].view(torch.int32), b[key].view(torch.int32)), key


READERS = {
    "tiles": lambda vsr, m, sc: vsr.raster(m, sc, binned=True),
    "statistics": lambda vsr, m, sc: vsr.raster(m, sc, stats=True),
    "bin": lambda vsr, m, sc: (vsr.bin(m, sc), vsr.raster(m, sc, binned=True))[1],
}


@pytest.mark.parametrize("T", [600, 20_000])
@pytest.mark.parametrize("reader", sorted(READERS))
def test_bins_hold_a_denser_view(vsr, reader, T):
    tris = torch.from_numpy(_half(T, 5)).cuda()
    m = vsr.Map(320, 240, 0.2, 0.9, 0.9, 60.0)
    sc = vsr.Scene(tris, _turned(np.pi))
    vsr.raster(m, sc)  # sized for a view of almost nothing
    sparse = sc.bin_pairs()
    for a in np.linspace(np.pi, 0.0, 9)[1:]:
        sc.update(tris, _turned(a))
        out = vsr.raster(m, sc)
    pairs = sc.bin_pairs()
    assert pairs > 2 * sparse + 8192 or T < 1000
    ref = vsr.raster_dense(m, sc)
    _equal(out, ref)
    _equal(READERS[reader](vsr, m, sc), ref)
    assert sc.bin_pairs() == pairs
    assert vsr.last_device_status() == 0


def test_pairs_of_a_shaded_frame(vsr):
    """The pair count of a shaded forward is that of its own view."""
    tris = torch.from_numpy(_half(5000, 6)).cuda()
    m = vsr.Map(200, 120, 0.2, 0.9, 0.9, 90.0)
    sc, frags = vsr.Scene(tris, _turned(0.3)), vsr.Frags()
    for q in range(3):
        vsr.raster_shaded(m, sc, frags)
        shaded = sc.bin_pairs()
        vsr.bin(m, sc)
        assert sc.bin_pairs() == shaded, q
        m.update(200, 120, 0.3, 0.8, 0.9, 60.0 + 40.0 * q)
        sc.update(tris, _turned(0.8 - 0.4 * q))
    # 24 x 16 pixels of 20,000 triangles: every tile's candidates are shared
    # between several CTAs
    tris = torch.from_numpy(_half(20_000, 7)).cuda()
    m, sc = vsr.Map(24, 16, 0.2, 0.9, 0.9, 90.0), vsr.Scene(tris, _turned(0.0))
    vsr.raster_shaded(m, sc, frags)
    shaded = sc.bin_pairs()
    vsr.bin(m, sc)
    assert sc.bin_pairs() == shaded
    assert vsr.last_device_status() == 0


def test_captured_binning_after_walked_frames(vsr):
    """A binning captured after frames that stored none, its replays, and the
    eager calls around them; the bins made room for this view before."""
    tris = torch.from_numpy(_half(8000, 8)).cuda()
    m = vsr.Map(200, 120, 0.2, 0.9, 0.9, 90.0)
    sc = vsr.Scene(tris, _turned(0.0))
    vsr.raster(m, sc)
    for a in (0.1, 0.2):
        sc.update(tris, _turned(a))
        vsr.raster(m, sc)
    ref = vsr.raster_dense(m, sc)
    out = {key: torch.zeros_like(ref[key]) for key in KEYS}
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        vsr.bin(m, sc)
        vsr.raster(m, sc, out=out, binned=True)
    for _ in range(3):
        vsr.bin(m, sc)
        _equal(vsr.raster(m, sc, binned=True), ref)
        g.replay()
        torch.cuda.synchronize()
        _equal(out, ref)
        _equal(vsr.raster_dense(m, sc), ref)
        _equal(vsr.raster(m, sc), ref)
    assert vsr.last_device_status() == 0


def test_eager_bins_after_a_capture_that_sized_none(vsr):
    """A capture between the walked frames and an eager binning sizes nothing:
    the eager one still holds the denser view."""
    tris = torch.from_numpy(_half(20_000, 9)).cuda()
    m = vsr.Map(320, 240, 0.2, 0.9, 0.9, 60.0)
    sc = vsr.Scene(tris, _turned(np.pi))
    out = vsr.raster(m, sc)  # sized for a view of almost nothing
    vsr.raster(m, sc, out=out, binned=True)  # what a captured binned raster allocates
    sparse = sc.bin_pairs()
    for a in np.linspace(np.pi, 0.0, 5)[1:]:
        sc.update(tris, _turned(a))
        vsr.raster(m, sc, out=out)
    assert sc.bin_pairs() > 2 * sparse + 8192
    ref = vsr.raster_dense(m, sc)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):  # (never launched: its bins are too small for this view)
        vsr.bin(m, sc)
    vsr.bin(m, sc)
    _equal(vsr.raster(m, sc, binned=True), ref)
    assert vsr.last_device_status() == 0
