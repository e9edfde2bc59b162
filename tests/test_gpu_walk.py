"""The raster that walks the triangle grid (every frame of a scene after the
first of its shape) and the stored bins of the same walk, bit for bit against
the dense reference (every pixel x every triangle), at the edges of their
rules: triangle counts around the direct / grid limit, tiles wider than the
range table, tiles with enough candidates to be shared between CTAs, caps of
every grid level and of the list, poles and the longitude seam, triangles
crowded into a few cells, and triangles culled at set-up."""
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


def _rotation(seed):
    q, r = np.linalg.qr(np.random.default_rng(seed).normal(size=(3, 3)))
    q = q * np.sign(np.diag(r))
    return q if np.linalg.det(q) > 0 else -q


def _towards(d):
    """A camera rotation whose -z, +y or +z axis is the world's +z."""
    return {"seam": np.diag([-1.0, 1.0, -1.0]), "pole": np.array([[1.0, 0, 0], [0, 0, 1], [0, -1, 0]]),
            "front": np.eye(3)}[d]


def _crowd(n, spread, seed):
    """n small triangles around world +z."""
    t = scenes.random_triangles(n, 2.0, 20.0, 0.01, seed).astype(np.float64)
    c = t.mean(axis=1, keepdims=True)
    rho = np.linalg.norm(c, axis=2, keepdims=True)
    rng = np.random.default_rng(seed)
    d = np.stack([rng.normal(0, spread, n), rng.normal(0, spread, n), np.ones(n)], 1)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return (t - c + rho * d[:, None, :]).astype(np.float32)


def _mixed(n, seed):
    """Caps of every level and of the list, and some culled triangles."""
    parts = [scenes.random_triangles(-(-n // 4), 1.0, 30.0, j, seed + q)
             for q, j in enumerate((0.004, 0.03, 0.12, 0.9))]
    t = np.concatenate(parts)[:n] if n < 4 else np.concatenate(parts)
    t = t[:n]
    if n > 8:
        t[3] = 0.0  # vertices at the eye
        t[5, 1] = t[5, 0]  # no area
    return t


CASES = [
    # W, H, k, l, s, omega, triangles, rotation
    (64, 48, 0.2, 0.9, 0.9, 120.0, lambda: np.zeros((0, 3, 3), np.float32), None),
    (33, 17, 0.2, 0.9, 0.9, 120.0, lambda: _mixed(1, 1), None),
    (160, 96, 0.3, 0.8, 0.9, 200.0, lambda: _mixed(257, 2), 3),
    (160, 96, 0.3, 0.8, 0.9, 200.0, lambda: _mixed(640, 2), 3),   # the last direct count
    (160, 96, 0.3, 0.8, 0.9, 200.0, lambda: _mixed(641, 2), 3),   # the first with a grid
    (251, 143, -0.4, 0.7, 0.8, 300.0, lambda: _mixed(6000, 4), 5),
    (40, 24, -0.2, 1.0, 1.0, 360.0, lambda: _mixed(5000, 6), 7),  # tiles of a radian and more
    (16, 16, 0.0, 1.0, 1.0, 360.0, lambda: _mixed(3000, 8), None),  # one tile, the whole sphere
    (320, 176, 0.5, 1.0, 1.0, 170.0, lambda: scenes.random_triangles(20000, 1.0, 40.0, 0.02, 9), "pole"),
    (320, 176, 0.5, 1.0, 1.0, 170.0, lambda: scenes.random_triangles(20000, 1.0, 40.0, 0.02, 9), "seam"),
    (96, 80, 0.0, 1.0, 1.0, 40.0, lambda: _crowd(12000, 0.05, 10), "front"),  # shared tiles, few of them
    (96, 80, 0.0, 1.0, 1.0, 8.0, lambda: _crowd(12000, 0.004, 11), "pole"),   # one cell
    (800, 608, 0.0, 1.0, 1.0, 60.0, lambda: np.concatenate([  # shared tiles among many: helpers after the tiles
        _crowd(6000, 0.02, 12), scenes.random_triangles(6000, 1.0, 40.0, 0.02, 13)]), "front"),
    # more tiles of many candidates than can be shared at a time
    (800, 608, 0.1, 0.9, 0.9, 170.0, lambda: scenes.random_triangles(6000, 1.0, 30.0, 0.9, 15), None),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_walk_equals_dense(vsr, case):
    W, H, k, l, s, om, tris, rot = CASES[case]
    M = None if rot is None else (_towards(rot) if isinstance(rot, str) else _rotation(rot))
    m = vsr.Map(W, H, k, l, s, om)
    sc = vsr.Scene(torch.from_numpy(tris()).cuda(), scenes.camera((0.0, 0.0, 0.0), M))
    ref = vsr.raster_dense(m, sc)
    first = vsr.raster(m, sc)               # stored bins, sized
    frames = [vsr.raster(m, sc) for _ in range(3)]  # the walk; the slots are reused
    pairs = sc.bin_pairs()
    bins = vsr.raster(m, sc, binned=True)   # the bins of the first frame
    vsr.bin(m, sc)
    assert vsr.last_device_status() == 0
    # the bins take the same triangles as the walk, tile by tile
    assert sc.bin_pairs() == pairs
    for out in [first, *frames, bins, vsr.raster(m, sc, binned=True)]:
        for key in ("id", "depth", "cov"):
            assert torch.equal(out[key].view(torch.int32), ref[key].view(torch.int32)), key


def test_tiles_after_an_unstored_frame(vsr):
    """vsr_raster_tiles after frames that stored no bins: for another lens
    and another set-up of a known shape."""
    tris = torch.from_numpy(scenes.random_triangles(3000, 1.0, 30.0, 0.05, 14)).cuda()
    m = vsr.Map(200, 120, 0.2, 0.9, 0.9, 150.0)
    sc = vsr.Scene(tris, scenes.camera())
    vsr.raster(m, sc)
    for q in range(2):
        m.update(200, 120, 0.3, 0.8, 0.9, 160.0 + 20.0 * q)
        sc.update(tris, scenes.camera((0.1 * q, 0.0, 0.1)))
        with pytest.raises(vsr.VsrError):
            vsr.raster(m, sc, binned=True)  # nothing binned or rasterized yet
        a = vsr.raster(m, sc)
        b = vsr.raster(m, sc, binned=True)
        for key in a:
            assert torch.equal(a[key].view(torch.int32), b[key].view(torch.int32)), key
    assert vsr.last_device_status() == 0


@pytest.mark.parametrize("T", [200, 5000])
def test_second_frame_under_capture(vsr, T):
    """The second frame of a shape is the first that walks: nothing is left
    for it to allocate, so it can be captured."""
    sc = vsr.Scene(torch.from_numpy(scenes.random_triangles(T, 1.0, 30.0, 0.05, 16)).cuda(), scenes.camera())
    m = vsr.Map(200, 120, 0.2, 0.9, 0.9, 150.0)
    first = vsr.raster(m, sc)
    out = {key: torch.empty_like(t) for key, t in first.items()}
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        vsr.raster(m, sc, out=out)
    for _ in range(3):
        for t in out.values():
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        for key in first:
            assert torch.equal(out[key].view(torch.int32), first[key].view(torch.int32)), key
    assert vsr.last_device_status() == 0
