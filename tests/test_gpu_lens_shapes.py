"""The lens tensor of render_shaded: four numbers, one a row, as a vector or a
column, of any floating type, on either side of the host link."""
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


@pytest.mark.parametrize("shape", [(4,), (4, 1)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("device", ["cpu", "cuda"])
def test_forward_takes_the_lens(vsr, shape, dtype, device):
    tris = torch.from_numpy(scenes.random_triangles(80, 1.0, 10.0, 0.25, 2)).cuda()
    colors = torch.ones(80, device="cuda")
    lens = torch.tensor([0.25, 0.75, 0.875, 160.0], dtype=dtype, device=device)
    r = vsr.ShadedRenderer(64, 48)
    ref = vsr.render_shaded(tris, colors, torch.tensor([0.25, 0.75, 0.875, 160.0], dtype=torch.float64), r)
    got = vsr.render_shaded(tris, colors, lens.reshape(shape), r)
    for a, b in zip(got, ref):
        assert torch.equal(a, b)
