"""The whole-frame global sort (Gaussians by depth, then entries by tile)
against the stage calls' sort of the entries themselves, over the shapes its
passes depend on: Gaussian counts around a 4096-word chunk, one tile to more
than 2^16 (one to three tile passes), equal depths, and overflow."""
import numpy as np
import pytest

from paper_2609_03613_gb300 import scenes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_03613_gb300 import tilegs as G  # noqa: E402


def stage_frame(sc, cam, tile):
    ctx = G.Context("global", tile_size=tile)
    ds = G.DeviceScene.from_numpy(sc)
    proj = ctx.project(ds, cam)
    isect, m_cap, m_dev, m = ctx.tile_intersect(proj, sc.n, cam)
    words, offsets, _ = ctx.sort_or_bin(proj, ds.scales, sc.n, cam, isect, m_cap, m_dev)
    return m, ctx.rasterize_fwd(proj, sc.n, cam, words, offsets)


@pytest.mark.parametrize("equal", [False, True])
@pytest.mark.parametrize("n,w,h,tile", [(1, 16, 16, 16), (31, 8, 8, 8), (4095, 100, 60, 16), (4096, 256, 256, 16),
                                        (4097, 257, 250, 16), (9000, 640, 400, 32), (30000, 1000, 700, 8),
                                        (3000, 2200, 1930, 8)])
def test_frame_sort_equals_entry_sort(n, w, h, tile, equal):
    sc = scenes.mixture_scene(n, 17, sh_degree=0)
    if equal:  # runs of Gaussians at one depth: the camera looks along z
        sc.means[:, 2] = np.round(sc.means[:, 2] * 8) / 8
    cam = scenes.hd_camera(width=w, height=h, f=0.6 * max(w, h))
    m, ref = stage_frame(sc, cam, tile)
    ctx = G.Context("global", tile_size=tile)
    out = ctx.render(G.DeviceScene.from_numpy(sc), cam)
    torch.cuda.synchronize()
    assert ctx.error() == 0 and ctx.last_entry_count() == m
    for a, b in zip(out, ref):
        assert torch.equal(a, b)


def test_frame_sort_overflow_then_room():
    sc = scenes.mixture_scene(20000, 18, sh_degree=0)
    cam = scenes.hd_camera(width=320, height=200, f=200.0)
    ds = G.DeviceScene.from_numpy(sc)
    m, ref = stage_frame(sc, cam, 16)
    ctx = G.Context("global")
    ctx.reserve(sc.n, m // 2, cam.width, cam.height)
    out = ctx.render(ds, cam, flags=G.RENDER_NO_SYNC)
    assert ctx.error() == 2  # capacity; the frame is empty
    assert float(out[1].abs().max().item()) == 0.0
    ctx.clear_error()
    out = ctx.render(ds, cam)  # reads M and grows
    assert ctx.error() == 0
    for a, b in zip(out, ref):
        assert torch.equal(a, b)
