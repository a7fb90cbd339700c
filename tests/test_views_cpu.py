"""The binding's views of the library's buffers and its camera record against
the library's own layout (offsets, sizes), field by field; short or strided
buffers are refused."""
import ctypes as C
import types

import numpy as np
import pytest
import torch

from paper_2609_03613_gb300 import tilegs as G

pytestmark = pytest.mark.skipif(not G.lib_available(), reason="libtilegs.so is not built")

FIELDS = [("xy_ab", 16, torch.float32, 4), ("c_o_z", 16, torch.float32, 4), ("rgb", 16, torch.float32, 4),
          ("rect", 8, torch.int32, 2), ("radius", 4, torch.int32, 1)]


@pytest.mark.parametrize("lead", [0, 256, 4])
@pytest.mark.parametrize("n", [0, 1, 15, 16, 17, 63, 64, 65, 1000])
def test_views_are_the_library_layout(n, lead):
    L = G.lib()
    buf = torch.arange(lead + int(L.gs_projected_bytes(n)) + 64, dtype=torch.int64).to(torch.uint8)[lead:]
    got = G.projected_fields(buf, n)
    for f, (k, b, dt, w) in enumerate(FIELDS):
        o = int(L.gs_projected_offset(n, f))
        assert G.projected_offsets(n)[f] == o
        want = buf[o:o + b * n].view(dt)
        want = want.view(n, w) if w > 1 else want
        assert got[k].shape == want.shape and got[k].stride() == want.stride() and got[k].dtype == dt
        assert n == 0 or got[k].data_ptr() == want.data_ptr()
        assert torch.equal(got[k].view(torch.int32), want.view(torch.int32))
    g = G.grad_fields(buf, n)
    for f, k in enumerate(("xy_ab", "c_o_z", "rgb")):
        o = int(L.gs_grad2d_offset(n, f))
        want = buf[o:o + 16 * n].view(torch.float32).view(n, 4)
        assert g[k].shape == want.shape and (n == 0 or g[k].data_ptr() == want.data_ptr())
    if n:
        for call, end in ((G.projected_fields, G.projected_offsets(n)[-1]), (G.grad_fields, int(L.gs_grad2d_offset(n, 2)) + 16 * n)):
            call(buf[:end], n)
            with pytest.raises(RuntimeError):
                call(buf[:end - 4], n)
            with pytest.raises(RuntimeError):
                call(torch.zeros(4 * end, dtype=torch.uint8)[::2], n)


@pytest.mark.parametrize("make", [lambda m: m, lambda m: m.astype(np.float64), lambda m: m.T.copy().T,
                                  lambda m: m.tolist(), lambda m: m.reshape(-1)])
def test_camera_record(make):
    m = np.random.default_rng(5).normal(0, 1, (4, 4)).astype(np.float32)
    cam = types.SimpleNamespace(viewmat=make(m), fx=1.5, fy=np.float32(2.5), cx=3, cy=4.25, width=np.int64(640), height=480,
                                near=0.01, far=1e10)
    c = G.gs_camera(cam)
    np.testing.assert_array_equal(np.array(c.viewmat[:], np.float32), m.reshape(-1))
    assert (c.fx, c.fy, c.cx, c.cy, c.width, c.height) == (1.5, 2.5, 3.0, 4.25, 640, 480)
    assert c.near_plane == C.c_float(0.01).value and c.far_plane == C.c_float(1e10).value
    cam.viewmat = m.reshape(-1)[:15]
    with pytest.raises((IndexError, ValueError)):
        G.gs_camera(cam)
