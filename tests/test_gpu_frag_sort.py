"""Long fragment lists of the shaded forward: closed shells around the eye in
random order, so that every pixel has about as many fragments as there are
shells, at and beyond the lengths that are sorted as they are found (8), by
their depths in shared memory (22 and 48) and where they are stored; coincident
shells, whose depths are equal and whose order is that of the triangles; tiles
with and without a list, and tiles shared between CTAs.  The image against the
FP64 oracle; the gradients against those of the same triangles in order of
their distance (the oracle has none here: at an edge that two triangles of a
shell share, their masks add up to exactly one, and which of them saturates the
pixel, and so takes no gradient, is up to the rounding)."""
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


def _shells(n, level, coincident, seed):
    """n icospheres, each turned its own way, their triangles shuffled; with
    `coincident`, every shell twice."""
    rng = np.random.default_rng(seed)
    base = scenes.icosphere(level, 1.0).astype(np.float64)
    parts = []
    for r in rng.permutation(n) + 3.0:
        q, u = np.linalg.qr(rng.normal(size=(3, 3)))
        parts.append((r * base) @ (q * np.sign(np.diag(u))).T)
    t = np.concatenate(parts * 2 if coincident else parts).astype(np.float32)
    return t[rng.permutation(len(t))]


# shells, subdivision level, coincident, W, H, omega
CASES = [(7, 0, False, 40, 24, 60.0), (9, 0, False, 40, 24, 60.0), (22, 0, False, 40, 24, 60.0),
         (24, 0, False, 40, 24, 60.0), (47, 0, False, 33, 17, 30.0), (52, 0, False, 33, 17, 30.0),
         (11, 0, True, 33, 17, 30.0), (26, 0, True, 33, 17, 30.0),
         (20, 2, False, 40, 24, 120.0), (24, 2, False, 40, 24, 120.0), (60, 1, False, 40, 24, 120.0),
         (12, 2, True, 40, 24, 120.0), (30, 2, True, 24, 16, 250.0)]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_long_lists(vsr, case):
    n, level, coincident, W, H, om = CASES[case]
    tris = _shells(n, level, coincident, case)
    T = len(tris)
    rng = np.random.default_rng(100 + case)
    cols = rng.uniform(0.2, 1.0, T).astype(np.float32)
    up = rng.normal(size=(H, W)).astype(np.float32)
    cam = scenes.camera()
    r = vsr.ShadedRenderer(W, H, cam=cam)
    r.set_lens(0.3, 0.8, 0.9, om)
    td, cd = torch.from_numpy(tris).cuda(), torch.from_numpy(cols).cuda()
    r.scene.update(td, r.cam)
    for _ in range(2):
        out = vsr.raster_shaded(r.map, r.scene, r.frags, cd)
    g = vsr.raster_backward(r.map, r.scene, r.frags, td, cd, out["id"], dimage=torch.from_numpy(up).cuda())
    assert vsr.last_device_status() == 0
    m64 = r.map.download().astype(np.float64)
    img = oracle.shade(m64, oracle.setup(tris, cam), cols.astype(np.float64))
    assert np.abs(out["image"].cpu().numpy() - img).max() <= 1e-5
    if coincident:
        return  # in another order another of two equal triangles comes first
    order = np.argsort(np.linalg.norm(tris.astype(np.float64).mean(axis=1), axis=1), kind="stable")
    to, co = torch.from_numpy(tris[order]).cuda(), torch.from_numpy(cols[order]).cuda()
    r.scene.update(to, r.cam)
    near = vsr.raster_shaded(r.map, r.scene, r.frags, co)
    assert torch.equal(near["depth"], out["depth"])
    gn = vsr.raster_backward(r.map, r.scene, r.frags, to, co, near["id"], dimage=torch.from_numpy(up).cuda())
    for key in ("dtris", "dcolors"):
        a, b = g[key].cpu().numpy()[order], gn[key].cpu().numpy()
        # sums by float atomics in an order that varies
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b), key
    assert torch.allclose(g["dlens"], gn["dlens"], rtol=1e-4, atol=1e-4 * float(gn["dlens"].abs().max()))
