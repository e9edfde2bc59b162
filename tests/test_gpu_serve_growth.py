"""Workspaces of the rendering server that grow while other slots are busy:
bursts of requests of mixed sizes on several slots, small pictures first, then
larger ones whose tiles hold many times the triangles of one work item.  Every
picture must be the one of the same request rendered alone, and of the dense
reference (every pixel x every triangle) where that is affordable."""
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


def _object(n, spread, seed):
    """n small triangles in directions around the world's +z axis."""
    t = scenes.random_triangles(n, 2.0, 20.0, 0.01, seed).astype(np.float64)
    c = t.mean(axis=1, keepdims=True)
    rng = np.random.default_rng(seed)
    d = np.stack([rng.normal(0, spread, n), rng.normal(0, spread, n), np.ones(n)], 1)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return (t - c + np.linalg.norm(c, axis=2, keepdims=True) * d[:, None, :]).astype(np.float32)


# by size: (W, H), lens; the small ones first
SIZES = [(96, 64), (320, 240), (1024, 512), (1600, 900)]


@pytest.mark.parametrize("seed", [0, 1, 2])
def test_growing_workspaces_beside_busy_slots(vsr, seed):
    rng = np.random.default_rng(seed)
    tris = [torch.from_numpy(_object(60_000, 0.15, 20 + seed)).cuda(),
            torch.from_numpy(scenes.random_triangles(200_000, 1.0, 40.0, 0.0192, 30 + seed)).cuda()]
    srv = vsr.Server(budget_bytes=20 << 30, slots=6)
    ids = [srv.add_scene(t) for t in tris]
    lenses = [dict(k=float(rng.uniform(-0.8, 0.8)), l=float(rng.uniform(0.6, 1.0)), s=float(rng.uniform(0.6, 1.0)),
                   omega=float(rng.uniform(90.0, 250.0))) for _ in range(5)]
    reqs = []
    for burst in range(3):
        # each burst: small pictures on every workspace, then ever larger ones,
        # two scenes in turn, all slots busy
        for W, H in SIZES[:2 + burst] * 3:
            for q in range(4):
                lens = dict(W=W, H=H, **lenses[int(rng.integers(5))])
                cam = scenes.camera(rng.uniform(-0.5, 0.5, 3))
                out = {"id": torch.empty((H, W), dtype=torch.int32, device="cuda"),
                       "depth": torch.empty((H, W), dtype=torch.float32, device="cuda"),
                       "cov": torch.empty((H, W), dtype=torch.float32, device="cuda")}
                reqs.append((q % 2, lens, cam, out))
    torch.cuda.synchronize()
    for at in range(0, len(reqs), 24):  # with a pause between, so that slots are taken anew
        tickets = [srv.submit(ids[s], lens, cam, out) for s, lens, cam, out in reqs[at:at + 24]]
        for t in tickets:
            assert srv.wait(t)["status"] == 0
    srv.close()
    dense = {0, 1, len(reqs) - 1}
    for q, (s, lens, cam, out) in enumerate(reqs):
        m = vsr.Map(lens["W"], lens["H"], lens["k"], lens["l"], lens["s"], lens["omega"])
        sc = vsr.Scene(tris[s], cam)
        refs = [vsr.raster(m, sc)]
        if q in dense:
            refs.append(vsr.raster_dense(m, sc))
        for ref in refs:
            for key in ("id", "depth", "cov"):
                assert torch.equal(out[key].view(torch.int32), ref[key].view(torch.int32)), (q, lens["W"], key)
    # the larger pictures had tiles of several work items
    m = vsr.Map(1024, 512, 0.2, 0.9, 0.9, 150.0)
    sc = vsr.Scene(tris[0], scenes.camera())
    vsr.bin(m, sc)
    assert sc.bin_pairs() > 512 * 8
    assert vsr.last_device_status() == 0
