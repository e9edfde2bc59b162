"""Errors that the kernels of the host path and of the server raise reach the
caller: the frame that raised one reports it, the next one is clean again.  The
error is raised from the host, in the status word that the kernels would raise
it in (the first member of either handle, mapped host memory), between frames."""
import ctypes

import numpy as np
import pytest

from paper_2003_10558_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TIMEOUT, FRAG_OVERFLOW = -6, -5


@pytest.fixture(scope="module")
def vsr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_10558_gb300 import build, vsr as V
    build.build()
    V.load()
    return V


def _word(handle):
    return ctypes.cast(handle, ctypes.POINTER(ctypes.POINTER(ctypes.c_int)))[0]


def test_render_host_reports_what_its_kernels_raise(vsr):
    tris = scenes.random_triangles(3000, 1.0, 30.0, 0.05, 1)
    m, sc = vsr.Map(160, 96, 0.2, 0.9, 0.9, 150.0), vsr.Scene()
    ref = vsr.render_host(m, sc, tris)
    word = _word(sc.h)
    for code in (TIMEOUT, FRAG_OVERFLOW):
        assert word[0] == 0
        word[0] = code
        with pytest.raises(vsr.VsrError) as e:
            vsr.render_host(m, sc, tris)
        assert e.value.code == code and word[0] == 0
        out = vsr.render_host(m, sc, tris)
        for key in ref:
            assert np.array_equal(out[key].view(np.uint32), ref[key].view(np.uint32)), key
        word[0] = code
        vsr.render_host_async(m, sc, tris)
        assert vsr.load().vsr_render_host_wait(sc.h) == code
        vsr.render_host_async(m, sc, tris)
        assert vsr.load().vsr_render_host_wait(sc.h) == 0
    assert vsr.last_device_status() == 0


def test_requests_report_what_their_kernels_raise(vsr):
    tris = torch.from_numpy(scenes.random_triangles(3000, 1.0, 30.0, 0.05, 1)).cuda()
    lens = dict(W=160, H=96, k=0.2, l=0.9, s=0.9, omega=150.0)
    out = {"id": torch.empty((96, 160), dtype=torch.int32, device="cuda")}
    srv = vsr.Server(budget_bytes=1 << 30, slots=1)
    sid = srv.add_scene(tris)
    status = []
    for code in (0, TIMEOUT, 0, FRAG_OVERFLOW, 0):
        _word(srv.h)[0] = code
        status.append(srv.wait(srv.submit(sid, lens, scenes.camera(), out))["status"])
    st = srv.stats()
    srv.close()
    assert status == [0, TIMEOUT, 0, FRAG_OVERFLOW, 0]
    assert st["completed"] == 3 and st["failed"] == 2
    assert vsr.last_device_status() == 0


def test_overflows_of_reruns_are_no_error(vsr):
    """A request whose bins overflow raises that in its slot's word from the
    device; rendered again, it is a success, and nothing is left behind."""
    tris = torch.from_numpy(scenes.random_triangles(12000, 1.0, 40.0, 0.02, 31)).cuda()
    srv = vsr.Server(budget_bytes=4 << 30, slots=1)
    sid = srv.add_scene(tris)
    for W, H in ((64, 48), (1024, 1024), (64, 48)):
        lens = dict(W=W, H=H, k=0.2, l=0.9, s=0.9, omega=250.0)
        out = {"id": torch.empty((H, W), dtype=torch.int32, device="cuda")}
        assert srv.wait(srv.submit(sid, lens, scenes.camera(), out))["status"] == 0
        assert _word(srv.h)[0] == 0
    assert srv.stats()["reruns"] >= 1
    srv.close()
    assert vsr.last_device_status() == 0
