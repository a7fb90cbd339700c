"""The forward raster where its work split can go wrong: images one pixel past
and one short of a warp's 8 x 8 block and of its two pixels a lane (x and
x + 4), frames on both sides of the rule that picks the round width (tiles
resident at once or not), and segments on both sides of a staging batch and of
the in-raster sort's buffer, against the oracle bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_2609_03613_gb300 import scenes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_03613_gb300 import tilegs as G  # noqa: E402


def assert_image(mode, sc, cam, tile, K, ref, **cfg):
    ctx = G.Context(mode, tile_size=tile, K=K, **cfg)
    rgb, alpha, last = (t.cpu().numpy() for t in ctx.render(G.DeviceScene.from_numpy(sc), cam, (0.1, 0.2, 0.3)))
    assert ctx.error() == 0
    np.testing.assert_array_equal(rgb.view(np.uint32), ref[0].view(np.uint32))
    np.testing.assert_array_equal(alpha.view(np.uint32), ref[1].view(np.uint32))
    np.testing.assert_array_equal(last, ref[2])


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("w,h", [(1, 1), (4, 7), (5, 8), (9, 17), (36, 33), (384, 304), (385, 304),
                                 (608, 768), (609, 768)])
def test_ragged_sizes_and_pixels_a_lane(w, h, tile):
    sc = scenes.mixture_scene(3000, 91)
    cam = scenes.hd_camera(width=w, height=h, f=max(w, h) * 0.6)
    ref = O.render(sc, cam, tile, bg=(0.1, 0.2, 0.3))[3]
    for mode in ("exact", "global"):
        assert_image(mode, sc, cam, tile, 64 if mode == "exact" else 1, ref)


@pytest.mark.parametrize("w,h", [(384, 608), (385, 608), (640, 608), (641, 608)])
def test_both_sides_of_the_rule(w, h):
    # 1520 tiles go by one pixel a lane, 1558 by two (the backward's line lies
    # between 912 and 950): the image, and the ends
    # of the 8 x 8 blocks that the backward starts from (it skips what lies
    # beyond, so a frame's gradients equal those of the stages, which walk on
    # to the tile's end, up to the order of their float32 atomics)
    sc = scenes.mixture_scene(60_000, 92)
    cam = scenes.hd_camera(width=w, height=h, f=400.0)
    ref = O.render(sc, cam, 16, bg=(0.1, 0.2, 0.3))[3]
    assert_image("exact", sc, cam, 16, 64, ref)
    dC, dA = (torch.from_numpy(x).cuda() for x in scenes.incoming_grads(h, w, seed=3))
    ds = G.DeviceScene.from_numpy(sc)
    ctx = G.Context("exact")
    kept = ctx.render(ds, cam, flags=G.RENDER_SAVE)  # the backward reads its last-id output
    got = G.grad_fields(ctx.render_bwd(dC, dA), sc.n)
    proj = ctx.project(ds, cam)
    isect, m_cap, m_dev, _ = ctx.tile_intersect(proj, sc.n, cam)
    words, offsets, _ = ctx.sort_or_bin(proj, ds.scales, sc.n, cam, isect, m_cap, m_dev)
    saved = ctx.rasterize_fwd(proj, sc.n, cam, words, offsets, save=True)[3]
    want = G.grad_fields(ctx.rasterize_bwd(proj, sc.n, cam, words, offsets, saved, dC, dA), sc.n)
    torch.cuda.synchronize()
    assert ctx.error() == 0
    del kept
    for k in got:
        np.testing.assert_allclose(got[k].cpu(), want[k].cpu(), rtol=1e-5, atol=1e-6 * float(want[k].abs().max()))


def one_tile(count, depths):
    """`count` Gaussians inside one tile, which stops after some two thousand."""
    rng = np.random.default_rng(count)
    cam = scenes.tiny_camera()
    z = rng.uniform(-0.4, 0.4, count)
    if depths == "equal":
        z = np.where(rng.random(count) < 0.7, 0.1, z)
    elif depths == "skewed":
        z = 0.4 - 0.8 * rng.random(count) ** 40
    xy = (132.0 + rng.uniform(-1.0, 1.0, (count, 2)) - cam.cx) * (3.0 - z)[:, None] / cam.fx
    return cam, scenes.Scene(np.column_stack([xy, z]).astype(np.float32), np.full((count, 3), 0.002, np.float32),
                             np.tile(np.array([1, 0, 0, 0], np.float32), (count, 1)),
                             np.full(count, 0.0045, np.float32), rng.uniform(0, 1, (count, 1, 3)).astype(np.float32), 0)


@pytest.mark.parametrize("depths", ["spread", "equal", "skewed"])
@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("count", [128, 129, 256, 257, 512, 513, 2048, 2049, 8191, 8192, 8193])
def test_segments_at_batch_and_sort_limits(count, tile, depths):
    # one bin a tile holding `count` entries: staged at rank, in depth buckets in
    # the raster, or sorted before it.  Equal depths and depths crowded at one
    # end fill a bucket past its limit.
    cam, sc = one_tile(count, depths)
    P, ent, (off, stream), ref = O.render(sc, cam, tile, bg=(0.1, 0.2, 0.3))
    assert np.diff(off).max() == count
    assert_image("exact", sc, cam, tile, 1, ref)


@pytest.mark.parametrize("depths", ["spread", "equal", "skewed"])
@pytest.mark.parametrize("count", [2, 32, 33, 128, 512, 513, 4096, 4097])
def test_segments_sorted_before_the_raster(count, depths):
    # the repair outside the raster: a segment sorted in registers, by a warp, by
    # a block (depth buckets; the network past a full bucket), or as a tail
    cam, sc = one_tile(count, depths)
    P, ent, (off, stream), ref = O.render(sc, cam, 16, bg=(0.1, 0.2, 0.3))
    assert np.diff(off).max() == count
    assert_image("exact", sc, cam, 16, 1, ref, repair_in_raster=0)
