"""A launch that the driver refuses fails its own call and no other: the error
is not found again by the next call's check."""
import ctypes
from types import SimpleNamespace

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


@pytest.mark.parametrize("T", [200, 2000])
def test_refused_launch_leaves_no_error(vsr, T):
    tris = torch.from_numpy(scenes.random_triangles(T, 1.0, 30.0, 0.1, 1)).cuda()
    m = vsr.Map(96, 64, 0.2, 0.9, 0.9, 150.0)
    sc, other = vsr.Scene(tris, scenes.camera()), vsr.Scene(tris, scenes.camera())
    ref = vsr.raster_dense(m, other)
    torch.cuda.synchronize()
    # no launch on the legacy stream while a stream that waits for it captures
    cu = ctypes.CDLL("libcuda.so.1")
    st, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert cu.cuStreamCreate(ctypes.byref(st), 0) == 0
    assert cu.cuStreamBeginCapture_v2(st, 0) == 0
    with pytest.raises(vsr.VsrError) as e:
        sc.update(tris, scenes.camera(), stream=SimpleNamespace(cuda_stream=0))
    cu.cuStreamEndCapture(st, ctypes.byref(graph))
    cu.cuStreamDestroy_v2(st)
    assert e.value.code == vsr.VSR_ERR_CUDA
    out = vsr.raster_dense(m, other)  # its launch is checked by the runtime's last error
    sc.update(tris, scenes.camera())
    again = vsr.raster(m, sc)
    for key in ref:
        assert torch.equal(out[key].view(torch.int32), ref[key].view(torch.int32)), key
        assert torch.equal(again[key].view(torch.int32), ref[key].view(torch.int32)), key
    assert vsr.last_device_status() == 0
