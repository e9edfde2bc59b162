"""The fragment lists of the shaded forward at the edges of their rules: tiles
at and beyond the triangle list the count pass keeps (128), pixels at and
beyond the length sorted in shared memory (8), tiles of more candidates than
one block of the walk; image, coverage and the gradients of a random upstream
against the FP64 oracle, ids and depths against the coverage path."""
import numpy as np
import pytest

import oracle
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


# W, H, triangles, jitter
CASES = [(33, 17, 1, 0.3), (48, 40, 40, 0.3), (40, 24, 128, 0.6), (40, 24, 129, 0.6), (37, 21, 700, 0.25),
         (24, 16, 3000, 0.08)]


@pytest.mark.parametrize("W,H,T,jitter", CASES)
def test_lists(vsr, W, H, T, jitter):
    k, l, s, om = 0.3, 0.8, 0.9, 200.0
    tris = scenes.random_triangles(T, 1.0, 10.0, jitter, seed=T)
    cols = np.random.default_rng(T).uniform(0.2, 1.0, T).astype(np.float32)
    up = np.random.default_rng(T + 1).normal(size=(H, W)).astype(np.float32)
    cam = scenes.camera()
    r = vsr.ShadedRenderer(W, H, cam=cam)
    eff = r.set_lens(k, l, s, om)
    td, cd = torch.from_numpy(tris).cuda(), torch.from_numpy(cols).cuda()
    r.scene.update(td, r.cam)
    ref = vsr.raster(r.map, r.scene)
    for _ in range(2):  # the second frame reuses lists and cursor
        out = vsr.raster_shaded(r.map, r.scene, r.frags, cd)
    g = vsr.raster_backward(r.map, r.scene, r.frags, td, cd, out["id"], dimage=torch.from_numpy(up).cuda())
    assert vsr.last_device_status() == 0
    for key in ("id", "depth"):
        assert torch.equal(out[key].view(torch.int32), ref[key].view(torch.int32)), key
    assert (out["cov"] - ref["cov"]).abs().max().item() <= 2e-6
    m64 = r.map.download().astype(np.float64)
    img = oracle.shade(m64, oracle.setup(tris, cam), cols.astype(np.float64))
    assert np.abs(out["image"].cpu().numpy() - img).max() <= 1e-5
    og = oracle.render_grad(m64, eff, tris.astype(np.float64), cols.astype(np.float64), up.ravel().astype(np.float64),
                            cam=np.asarray(cam, dtype=np.float64))
    for a, b in ((g["dtris"], og["dtris"]), (g["dcolors"], og["dcolors"])):
        assert np.linalg.norm(a.cpu().numpy() - b) <= 1e-3 * np.linalg.norm(b)


@pytest.mark.parametrize("n", [1, 2, 5])
def test_lists_grow(vsr, n):
    """Frames of ever more fragments into lists filled before their number is
    known: the same as into lists of their own, and no error."""
    m = vsr.Map(61, 45, 0.3, 0.8, 0.9, 200.0)
    frags = vsr.Frags()
    for q in range(3):
        sc = vsr.Scene(torch.from_numpy(scenes.random_triangles(20 * (4 * n) ** q, 1.0, 10.0, 0.2, seed=q)).cuda(),
                       scenes.camera())
        out, ref = (vsr.raster_shaded(m, sc, f) for f in (frags, vsr.Frags()))
        for key in ref:
            assert torch.equal(out[key].view(torch.int32), ref[key].view(torch.int32)), key
    assert vsr.last_device_status() == 0
