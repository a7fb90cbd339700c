"""The depth-range selection at its limits: sample counts around the cap and
around a warp, keys that differ in their last bits, in two values, in none, or
over many binades (one to three radix passes), against the oracle bit for bit;
and a whole frame's sampled keys, which are taken from the Gaussians' entry
offsets instead of the entries, against the stages'."""
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


def points(depth):
    """One Gaussian of one tile at each depth along a ray of the tiny camera."""
    cam = scenes.tiny_camera()
    n = depth.shape[0]
    m = np.zeros((n, 3), np.float32)
    m[:, 2] = 3.0 - depth
    m[:, :2] = (np.array([132.0 - cam.cx, 132.0 - cam.cy]) * depth[:, None] / cam.fx)
    return cam, scenes.Scene(m, np.tile((1e-4 * depth[:, None]).astype(np.float32), (1, 3)),
                             np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1)), np.full(n, 0.5, np.float32),
                             np.full((n, 1, 3), 0.3, np.float32), 0)


@pytest.mark.parametrize("keys", ["spread", "equal", "two", "last_bits", "binades"])
@pytest.mark.parametrize("n", [1, 2, 33, 100, 8191, 8192, 8193, 30000])
def test_order_statistics(n, keys):
    rng = np.random.default_rng(n)
    if keys == "spread":
        z = rng.uniform(1.0, 5.0, n)
    elif keys == "equal":
        z = np.full(n, 3.0)
    elif keys == "two":
        z = np.where(rng.random(n) < 0.985, 2.0, 4.0)
    elif keys == "last_bits":
        z = 3.0 - rng.integers(0, 5, n) * 2.0 ** -22
    else:
        z = 10.0 ** rng.uniform(-1.0, 6.0, n)
    cam, sc = points(z)
    P = O.project(sc, cam)
    ent = O.emit(P, cam.width, cam.height)
    assert ent[0].shape[0] > 0
    for mode in ("exact", "paper"):
        ctx = G.Context(mode)
        ds = G.DeviceScene.from_numpy(sc)
        proj = ctx.project(ds, cam)
        isect, m_cap, m_dev, _ = ctx.tile_intersect(proj, sc.n, cam)
        zr = ctx.depth_range(proj, ds.scales, sc.n, cam, isect, m_cap, m_dev).cpu().numpy()
        want, _ = O.depth_range(ent[2], P["depth"], sc.scales, near_shift=mode == "paper")
        np.testing.assert_array_equal(zr.view(np.uint32), np.asarray(want, np.float32).view(np.uint32))


@pytest.mark.parametrize("n", [1, 61, 255, 1021, 4098, 30000, 400000])
def test_frame_samples(n):
    # a frame's planned bins and so the tiles its first pass leaves unfinished
    # follow from its bin splits: the same tiles as the stages', whose range is
    # the oracle's
    sc = scenes.mixture_scene(n, 12)
    cam = scenes.hd_camera(width=517, height=301, f=320.0)
    w = torch.from_numpy(_bias_only(1))
    ctx = G.Context("exact", planner=1)
    ctx.set_planner_weights(w)
    ds = G.DeviceScene.from_numpy(sc)
    ctx.render(ds, cam)
    torch.cuda.synchronize()
    st = G.Context("exact", planner=1)
    st.set_planner_weights(w)
    proj = st.project(ds, cam)
    isect, m_cap, m_dev, m = st.tile_intersect(proj, sc.n, cam)
    zr = st.depth_range(proj, ds.scales, sc.n, cam, isect, m_cap, m_dev)
    P = O.project(sc, cam)
    want, _ = O.depth_range(O.emit(P, cam.width, cam.height)[2], P["depth"], sc.scales, near_shift=False)
    np.testing.assert_array_equal(zr.cpu().numpy().view(np.uint32), np.asarray(want, np.float32).view(np.uint32))
    words, offsets, _ = st.sort_or_bin(proj, ds.scales, sc.n, cam, isect, m_cap, m_dev)
    plan, _ = st.plan_tiles(cam, offsets)
    flags = st.rasterize_fwd_plan(proj, sc.n, cam, words, offsets, plan=plan, flags=True)[3]
    assert ctx.flagged_tiles() == int(flags.sum())
    assert n < 30000 or ctx.flagged_tiles() > 0
