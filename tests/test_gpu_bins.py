"""Bin construction where its row spans and counts can go wrong: one to nine tile
rows and columns (spans that end on the grid's last column, windows of 32
records that start and end inside a Gaussian), grids on both sides of the
one-pass offsets, a planned frame's completing pass and a batch of such views:
the oracle's image bit for bit, or the single frames'."""
import numpy as np
import pytest

import oracle as O
from paper_2609_03613_gb300 import scenes
from test_gpu_planner import _bias_only

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_03613_gb300 import tilegs as G  # noqa: E402

BG = (0.1, 0.2, 0.3)


def assert_same(out, ref):
    for a, b in zip(out, ref):
        np.testing.assert_array_equal(a.cpu().numpy().view(np.uint32), np.asarray(b).view(np.uint32))


@pytest.mark.parametrize("planner", [0, 1])
@pytest.mark.parametrize("tile,K", [(16, 64), (8, 128), (32, 1)])
@pytest.mark.parametrize("tx,ty", [(1, 1), (2, 2), (3, 3), (5, 4), (8, 5), (7, 7), (9, 8), (2, 9)])
def test_small_grids(tx, ty, tile, K, planner):
    sc = scenes.mixture_scene(2500, 7 * tx + ty)
    cam = scenes.hd_camera(width=tile * tx - 3, height=tile * ty - 1, f=tile * max(tx, ty) * 0.5)
    ctx = G.Context("exact", tile_size=tile, K=K, planner=planner)
    if planner:
        ctx.set_planner_weights(torch.from_numpy(_bias_only(0)))
    out = ctx.render(G.DeviceScene.from_numpy(sc), cam, BG)
    assert ctx.error() == 0
    assert_same(out, O.render(sc, cam, tile, bg=BG)[3])


@pytest.mark.parametrize("planner", [0, 1])
@pytest.mark.parametrize("w,h", [(5088, 33), (5104, 81)])
def test_both_sides_of_the_one_pass_offsets(w, h, planner):
    # 318 tiles of 129 words a row fill the offsets' shared memory, 319 do not
    sc = scenes.mixture_scene(4000, 3)
    cam = scenes.hd_camera(width=w, height=h, f=900.0)
    ctx = G.Context("exact", K=128, planner=planner)
    if planner:
        ctx.set_planner_weights(torch.from_numpy(_bias_only(0)))
    out = ctx.render(G.DeviceScene.from_numpy(sc), cam, BG)
    assert ctx.error() == 0
    assert_same(out, O.render(sc, cam, 16, bg=BG)[3])


@pytest.mark.parametrize("K", [64, 128])
def test_batch_of_uneven_grids(K):
    sc = G.DeviceScene.from_numpy(scenes.mixture_scene(6000, 5))
    cams = [scenes.hd_camera(width=w, height=h, f=max(w, h) * 0.6)
            for w, h in [(16, 16), (33, 40), (70, 95), (129, 64), (50, 130), (5104, 40)]]
    single = G.Context("exact", K=K)
    batch = G.Context("exact", K=K)
    for views in (cams[:5], cams):  # one-pass offsets; the last view's rows too wide for them at K = 128
        outs = batch.render_batch(sc, views, bg=BG)
        torch.cuda.synchronize()
        assert batch.error() == 0
        for cam, out in zip(views, outs):
            assert_same(out, [t.cpu().numpy() for t in single.render(sc, cam, BG)])
