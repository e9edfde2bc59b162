"""Gradients when some of the backward calls are captured in CUDA graphs and
others run eagerly, in any order: each call's gradients are those of a forward
and backward on their own."""
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


class Step:
    """A forward's state; back() runs the adjoint for `want`."""

    def __init__(self, vsr):
        W, H, T = 96, 64, 700
        self.vsr = vsr
        self.m = vsr.Map(W, H, 0.3, 0.8, 0.9, 170.0)
        self.tris = torch.from_numpy(scenes.random_triangles(T, 1.0, 10.0, 0.15, 3)).cuda()
        self.colors = torch.from_numpy(np.random.default_rng(4).uniform(0.2, 1.0, T).astype(np.float32)).cuda()
        self.up = torch.from_numpy(np.random.default_rng(5).normal(size=(H, W)).astype(np.float32)).cuda()
        self.sc, self.frags = vsr.Scene(self.tris, scenes.camera()), vsr.Frags()
        self.out = vsr.raster_shaded(self.m, self.sc, self.frags, self.colors)

    def back(self, *want):
        return self.vsr.raster_backward(self.m, self.sc, self.frags, self.tris, self.colors, self.out["id"],
                                        dimage=self.up, want=want)

    def capture(self, *want):
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            out = self.back(*want)
        return g, out


ALL = ("tris", "colors", "lens")


def _same(a, ref):
    torch.cuda.synchronize()
    for key in a:
        # sums by float atomics in an order that varies
        assert (a[key] - ref[key]).norm() <= 1e-4 * ref[key].norm(), key


@pytest.mark.parametrize("leftover", [("lens",), ("tris",), ALL])
def test_eager_backward_between_capture_and_replay(vsr, leftover):
    ref = Step(vsr).back(*ALL)
    s = Step(vsr)
    _same(s.back(*ALL), ref)
    _same(s.back(*leftover), ref)
    g, out = s.capture(*ALL)
    _same(s.back(*ALL), ref)  # before the first replay
    for _ in range(2):
        g.replay()
        _same(out, ref)
    _same(s.back(*ALL), ref)
    assert vsr.last_device_status() == 0


def test_replayed_lens_backward_beside_eager_ones(vsr):
    ref = Step(vsr).back(*ALL)
    s = Step(vsr)
    _same(s.back(*ALL), ref)
    g, out = s.capture("lens")
    for _ in range(3):
        _same(s.back(*ALL), ref)
        g.replay()
        _same(out, ref)
        _same(s.back("colors"), ref)
        g.replay()
    _same(s.back(*ALL), ref)
    assert vsr.last_device_status() == 0
