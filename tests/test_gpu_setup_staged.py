"""Set-up from vertices staged in whole lines (pinned host memory, batches):
triangle counts around a CTA's 256 and 16-byte-aligned and unaligned buffers,
bit for bit against the set-up that reads a device buffer in place."""
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


@pytest.mark.parametrize("skip", [0, 1])
@pytest.mark.parametrize("T", [1, 2, 255, 256, 257, 1031])
@pytest.mark.parametrize("rotated", [False, True])
def test_staged_equals_in_place(vsr, T, skip, rotated):
    tris = scenes.random_triangles(T, 1.0, 10.0, 0.3, seed=T)
    rot = np.array([[0.0, 1, 0], [0, 0, 1], [1, 0, 0]]) if rotated else None
    cam = scenes.camera((0.1, 0.0, -0.2), rot)
    W, H = 72, 40
    m = vsr.Map(W, H, 0.3, 0.8, 0.9, 200.0)
    ref = vsr.raster(m, vsr.Scene(torch.from_numpy(tris).cuda(), cam))
    pinned = torch.empty(9 * T + skip).pin_memory()
    pinned[skip:] = torch.from_numpy(tris.ravel())
    outs = [vsr.render_host(m, vsr.Scene(), pinned.numpy()[skip:].reshape(T, 3, 3), cam)]
    dev = torch.empty(9 * T + skip, device="cuda")
    dev[skip:] = pinned[skip:].cuda()
    out = {k: torch.empty((H, W), dtype=t, device="cuda")
           for k, t in (("id", torch.int32), ("depth", torch.float32), ("cov", torch.float32))}
    vsr.Batch().render([m], dev[skip:].view(T, 3, 3), [cam], [out])
    outs.append({k: v.cpu().numpy() for k, v in out.items()})
    for o in outs:
        for key in ("id", "depth", "cov"):
            assert np.array_equal(o[key].view(np.uint32), ref[key].cpu().numpy().view(np.uint32)), key
