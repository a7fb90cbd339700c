"""The framework's performance cases: what a user's program has it do, called
through its public entry points (tilegs.Context, autograd.rasterize and the
planner's training kernels).

A case is a dict of plain values.  Its `path` says which calls it makes:

  view     one camera's frame of a resident scene (Context.render), as a viewer
           or an evaluation loop renders it
  train    a training step on a whole frame: Context.render with RENDER_SAVE,
           then Context.render_bwd
  stages   a training step through the stage calls and the autograd function,
           as a program that needs the projected record itself writes it
  batch    several cameras of one scene in one call (Context.render_batch)
  fit      one optimiser step of the bin planner's network

Scenes are drawn on the GPU with the distributions of
paper_2609_03613_gb300/scenes.py: "plain" (uniform means, degree-0 colour, like
tiny_scene) and "mixture" (64 anisotropic clusters and a shell, like
mixture_scene).  A "deep" camera stands inside a cluster (like heavy_camera),
the others on a sphere around the scene (like batch_cameras).
"""
import math
import os

import numpy as np
import torch

from paper_2609_03613_gb300 import autograd as GA
from paper_2609_03613_gb300 import scenes
from paper_2609_03613_gb300 import tilegs as G

_ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_WEIGHTS = os.path.join(_ROOT, "paper_2609_03613_gb300", "planner_weights.npy")
_BG = (0.1, 0.2, 0.3)


# ---------------------------------------------------------------- the cases
def _case(path, n, w=0, h=0, deg=3, mode="exact", tile=16, K=64, scene="mixture", deep=False, planner=False,
          graph=False, host=False, views=1):
    return {"path": path, "n": n, "w": w, "h": h, "deg": deg, "mode": mode, "tile": tile, "K": K, "scene": scene,
            "deep": deep, "planner": planner, "graph": graph, "host": host, "views": views}


def listed():
    return [
        # a thumbnail of a small object: the smallest call, launches and latency
        dict(_case("view", 10_000, 256, 256, deg=0, scene="plain"), name="view_tiny"),
        # a small preview with odd sizes and the autotuner's smallest tile
        dict(_case("view", 40_003, 501, 333, deg=1, tile=8), name="view_preview_tile8"),
        # the ordinary frame of a viewer or benchmark: 1M Gaussians at 1080p, replayed as a graph
        dict(_case("view", 1_000_000, 1920, 1080, graph=True), name="view_1080p_graph"),
        # a rendering service: odd sizes, launched call by call, the image fetched to the host
        dict(_case("view", 437_501, 1237, 823, deg=2, host=True), name="view_odd_host"),
        # a walk through a large scene: the camera inside a dense cluster, thousands of entries a tile
        dict(_case("view", 3_000_000, 1920, 1080, deep=True), name="view_deep_1080p"),
        # the same at a higher resolution with the learned bin planner, its deep-frame setting
        dict(_case("view", 4_000_000, 2560, 1440, deep=True, planner=True, graph=True), name="view_deep_1440p_planned"),
        # the global-sort path, which the method's users compare against and fall back to
        dict(_case("view", 500_000, 1280, 720, mode="global"), name="view_global_720p"),
        # the published method's own policy: near-shifted bins, rules and budget
        dict(_case("view", 300_000, 1280, 720, deg=2, mode="paper"), name="view_paper_720p"),
        # a training step on a full frame: forward saved for the backward, backward
        dict(_case("train", 1_000_000, 1920, 1080, graph=True), name="train_1080p"),
        # early training, stage by stage through autograd at a reduced, odd resolution
        dict(_case("stages", 120_007, 499, 285), name="train_stages_small"),
        # an evaluation set: sixteen cameras of uneven resolutions in one call
        dict(_case("batch", 1_000_000, graph=True, views=16), name="batch_16_views"),
        # one optimiser step of the bin planner's network on a minibatch of tiles
        dict(_case("fit", 4096), name="planner_fit_4096"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "view", "view", "deep", "train", "stages", "batch", "fit"])
    if kind == "view":
        mode = rng.choice(["exact", "exact", "exact", "global", "paper"])
        n = _log(rng, 5_000, 1_500_000 if mode == "exact" else 500_000)
        plain = n < 60_000 and rng.random() < 0.5
        return _case("view", n, _log(rng, 97, 1920), _log(rng, 97, 1080), deg=0 if plain else rng.randint(0, 3), mode=mode,
                     tile=rng.choice([16, 16, 16, 16, 8, 32]), K=rng.choice([64, 64, 64, 32, 128]),
                     scene="plain" if plain else "mixture", graph=rng.random() < 0.4, host=rng.random() < 0.15)
    if kind == "deep":
        planner = rng.random() < 0.5
        return _case("view", rng.randint(1_000_000, 3_000_000), rng.randint(1100, 1920), rng.randint(700, 1080), deep=True,
                     planner=planner, graph=planner)
    if kind == "train":
        return _case("train", _log(rng, 20_000, 1_000_000), _log(rng, 200, 1920), _log(rng, 200, 1080), deg=rng.randint(0, 3),
                     tile=rng.choice([16, 16, 16, 8, 32]), graph=rng.random() < 0.7)
    if kind == "stages":
        return _case("stages", _log(rng, 20_000, 300_000), _log(rng, 97, 900), _log(rng, 97, 700), deg=rng.randint(0, 3),
                     mode=rng.choice(["exact", "exact", "global"]))
    if kind == "batch":
        return _case("batch", _log(rng, 50_000, 1_000_000), deg=rng.randint(0, 3), graph=rng.random() < 0.7,
                     views=rng.randint(2, 12))
    return _case("fit", _log(rng, 500, 8192))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1009 + 17)


def _scene(case, seed):
    """(DeviceScene, cluster centres [64, 3] numpy or None), drawn on the GPU from the seed."""
    n, deg, g = case["n"], case["deg"], _gen(seed)
    nc = (deg + 1) ** 2
    normal = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    uniform = lambda *s: torch.rand(*s, generator=g, device="cuda")  # noqa: E731
    unit = lambda q: q / q.norm(dim=1, keepdim=True)  # noqa: E731
    centres = None
    if case["scene"] == "plain":
        means = uniform(n, 3) * 2 - 1
        scales = torch.exp(normal(n, 3) * 0.5 - 4.0)
        opac = torch.sigmoid(normal(n))
    else:
        c = uniform(64, 3) * 2 - 1
        sig = 0.05 + 0.25 * uniform(64, 3)
        rot = torch.linalg.qr(normal(64, 3, 3).cpu())[0].cuda()
        comp = torch.randint(0, 64, (n,), generator=g, device="cuda")
        mix = c[comp] + torch.einsum("nij,nj->ni", rot[comp], normal(n, 3) * sig[comp])
        shell = unit(normal(n, 3)) * (8 + 2 * uniform(n, 1))
        means = torch.where(uniform(n, 1) < 0.1, shell, mix)
        scales = torch.exp(normal(n, 3) - 5.0)
        opac = torch.sigmoid(1.5 * normal(n))
        centres = c.cpu().numpy().astype(np.float64)
    quats = unit(normal(n, 4))
    if deg == 0:
        sh = (uniform(n, 1, 3) * 2 - 1) * math.sqrt(math.pi)
    else:
        sh = 0.3 * normal(n, nc, 3)
    return G.DeviceScene(means.contiguous(), scales.contiguous(), quats.contiguous(), opac.contiguous(), sh.contiguous(),
                         deg), centres


def _cameras(case, seed, centres):
    rng = np.random.Generator(np.random.PCG64(int(seed) + 71))
    cams = []
    for _ in range(case["views"]):
        w, h = case["w"], case["h"]
        if case["path"] == "batch":
            w, h = scenes.BATCH_RESOLUTIONS[len(cams) % len(scenes.BATCH_RESOLUTIONS)]
        f = w * (1100.0 / 1920.0) if case["scene"] == "mixture" else float(w)
        if case["deep"]:
            pos = centres[int(rng.integers(0, 64))] + 0.05 * rng.standard_normal(3)
            if np.linalg.norm(pos) < 0.2:
                pos = pos + np.array([0.0, 0.0, 0.5])
        else:
            d = rng.standard_normal(3)
            pos = d / np.linalg.norm(d) * rng.uniform(2.5, 4.0)
        cams.append(scenes.Camera(scenes.look_at(pos), f, f, w / 2.0, h / 2.0, w, h))
    return cams


def _images(cam, host=False, last=True):
    at = dict(pin_memory=True) if host else dict(device="cuda")
    return (torch.empty((cam.height, cam.width, 3), **at), torch.empty((cam.height, cam.width), **at),
            torch.empty((cam.height, cam.width), dtype=torch.int32, **at) if last else None)


def _upstream(cam, seed):
    g = _gen(seed + 5)
    return (torch.randn((cam.height, cam.width, 3), generator=g, device="cuda"),
            torch.randn((cam.height, cam.width), generator=g, device="cuda"))


def _fit_inputs(case, seed):
    """A minibatch of standardised tile statistics with labels that depend on them, and fresh parameters."""
    g, B, F, H, C = _gen(seed), case["n"], G.PLAN_FEATURES, G.PLAN_HIDDEN, G.PLAN_CLASSES
    X = torch.randn(B, F, generator=g, device="cuda")
    y = (X[:, 0] * 1.5 + 0.5 * torch.randn(B, generator=g, device="cuda") + 2.5).round().clamp(0, C - 1).to(torch.int32)
    w = lambda n, s: torch.randn(n, generator=g, device="cuda") * s  # noqa: E731
    z = lambda n: torch.zeros(n, device="cuda")  # noqa: E731
    P = torch.cat([w(H * F, math.sqrt(2 / F)), z(H), w(H * H, math.sqrt(2 / H)), z(H), w(C * H, math.sqrt(1 / H)), z(C)])
    return X, y, P


def prepare(case, seed):
    path = case["path"]
    if path == "fit":
        X, y, P = _fit_inputs(case, seed)
        return {"case": case, "X": X, "y": y, "P": P, "m": torch.zeros_like(P), "v": torch.zeros_like(P), "step": 0}
    sc, centres = _scene(case, seed)
    cams = _cameras(case, seed, centres)
    cam = cams[0]
    ctx = G.Context(case["mode"], tile_size=case["tile"], K=case["K"], planner=1 if case["planner"] else 0)
    s = {"case": case, "sc": sc, "cams": cams, "ctx": ctx, "stream": torch.cuda.Stream() if case["graph"] else None}
    if case["planner"]:
        ctx.set_planner_weights(torch.from_numpy(np.load(_WEIGHTS)).cuda())
    if path == "batch":
        s["outs"] = [_images(c) for c in cams]
        ctx.render_batch(sc, cams, bg=_BG, outs=s["outs"])  # sizes every view's scratch
    elif path in ("view", "train"):
        # what a program does at start-up: one frame sizes the scratch, and the
        # entry capacity is reserved with some room
        s["out"] = _images(cam, case["host"], last=case["mode"] != "paper")  # an approximate frame has no use for ids
        ctx.render(sc, cam, bg=_BG, out=s["out"], flags=G.RENDER_HOST_OUTPUTS if case["host"] else 0)
        torch.cuda.synchronize()
        ctx.reserve(sc.n, int(ctx.last_entry_count() * 1.05) + 1024, cam.width, cam.height)
    if path == "train":
        s["up"] = _upstream(cam, seed)
        s["grad"] = torch.empty(int(G.lib().gs_grad2d_bytes(sc.n)), dtype=torch.uint8, device="cuda")
    if path == "stages":
        s["up"] = _upstream(cam, seed)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- one pass
def _view(s):
    case = s["case"]
    flags = (G.RENDER_GRAPH | G.RENDER_NO_SYNC) if case["graph"] and not case["host"] else 0
    if case["host"]:
        flags |= G.RENDER_HOST_OUTPUTS
    return s["ctx"].render(s["sc"], s["cams"][0], bg=_BG, out=s["out"], flags=flags)


def _train(s):
    flags = G.RENDER_SAVE | ((G.RENDER_GRAPH | G.RENDER_NO_SYNC) if s["case"]["graph"] else 0)
    out = s["ctx"].render(s["sc"], s["cams"][0], bg=_BG, out=s["out"], flags=flags)
    grad = s["ctx"].render_bwd(s["up"][0], s["up"][1], grad=s["grad"])
    f = G.grad_fields(grad, s["sc"].n)
    return list(out) + [f["xy_ab"], f["c_o_z"], f["rgb"]]


def _stages(s):
    ctx, sc, cam = s["ctx"], s["sc"], s["cams"][0]
    proj = ctx.project(sc, cam)
    isect, m_cap, m_dev, _ = ctx.tile_intersect(proj, sc.n, cam)
    words, offsets, _ = ctx.sort_or_bin(proj, sc.scales, sc.n, cam, isect, m_cap, m_dev)
    f = G.projected_fields(proj, sc.n)
    leaves = [f[k].detach().requires_grad_() for k in ("xy_ab", "c_o_z", "rgb")]
    frame = GA.Frame(ctx, proj, sc.n, cam, words, offsets, ctx.stride, _BG)
    img, alpha = GA.rasterize(*leaves, frame)
    torch.autograd.backward([img, alpha], list(s["up"]))
    return [img.detach(), alpha.detach()] + [t.grad for t in leaves]


def _fit(s):
    s["step"] += 1
    acts, logits = G.mlp_forward(s["P"], s["X"])
    loss, dz = G.mlp_loss_grad(logits, s["y"])
    grads = G.mlp_backward(s["P"], s["X"], acts, dz)
    G.adam_step(s["P"], grads, s["m"], s["v"], s["step"], 3e-3)
    return [loss, logits, grads, s["P"], s["m"], s["v"]]


def run(state):
    path = state["case"]["path"]
    if path == "fit":
        return _fit(state)
    call = {"view": _view, "train": _train, "stages": _stages}.get(path)
    if state["stream"] is not None:
        with torch.cuda.stream(state["stream"]):
            if path == "batch":
                return state["ctx"].render_batch(state["sc"], state["cams"], bg=_BG, outs=state["outs"],
                                                 flags=G.RENDER_GRAPH | G.RENDER_NO_SYNC)
            return call(state)
    if path == "batch":
        return state["ctx"].render_batch(state["sc"], state["cams"], bg=_BG, outs=state["outs"])
    return call(state)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: the scene (and upstream gradients) read once, the images (and
    gradients) written once.  Operations: ~400 a Gaussian and view for the
    projection and colour, and 60 pixel tests a pixel (the mean of the 1080p
    frame of 1M Gaussians) of 30 operations each, three times that with the
    backward; the network's products for a planner step."""
    n = case["n"]
    if case["path"] == "fit":
        F, H, C = G.PLAN_FEATURES, G.PLAN_HIDDEN, G.PLAN_CLASSES
        return {"bytes": 4 * (n * (F + 1 + C) + 7 * G.PLAN_PARAMS), "flops": 6 * n * (F * H + H * H + H * C)}
    scene = 4 * n * (11 + 3 * (case["deg"] + 1) ** 2)
    if case["path"] == "batch":
        sizes = [scenes.BATCH_RESOLUTIONS[i % len(scenes.BATCH_RESOLUTIONS)] for i in range(case["views"])]
        px = sum(w * h for w, h in sizes)
    else:
        px = case["w"] * case["h"]
    b, f = scene + 20 * px, 400 * n * case["views"] + 60 * 30 * px
    if case["path"] in ("train", "stages"):
        b, f = b + 16 * px + 48 * n, f + 2 * 60 * 30 * px
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times what was measured between the float32 frame and the
    64-bit one (exact): rounding moves an alpha test or a stop here and there
    and shifts transmittances deep in a pixel's list (images 3e-5; gradients of
    a full frame 2.3e-3, of a small one 5e-5).  Ids of the last Gaussian differ
    where a stop moves.  The paper policy leaves the order inside an
    unselected bin open, so its frames differ from run to run (7e-3 to 9e-3)."""
    if case["path"] == "fit":
        return {"rel": 1e-5, "max": 1e-2}
    if case["mode"] == "paper":
        return {"rel": 2.8e-2, "max": 0.95}
    if case["path"] == "train":
        return {"rel": 8e-3, "max": 0.5, "differ": 1e-3}
    if case["path"] == "stages":
        return {"rel": 2e-4, "max": 0.1}
    return {"rel": 1.2e-4, "max": 0.1, "differ": 1e-3}


# ---------------------------------------------------------------- the same in 64 bits
def _sh_basis(d):
    x, y, z = d.unbind(1)
    xx, yy, zz = x * x, y * y, z * z
    a1 = math.sqrt(3 / (4 * math.pi))
    a2, a20, a22 = math.sqrt(15 / math.pi) / 2, math.sqrt(5 / math.pi) / 4, math.sqrt(15 / math.pi) / 4
    a33, a32 = math.sqrt(35 / (2 * math.pi)) / 4, math.sqrt(105 / math.pi) / 2
    a31, a30, a34 = math.sqrt(21 / (2 * math.pi)) / 4, math.sqrt(7 / math.pi) / 4, math.sqrt(105 / math.pi) / 4
    return torch.stack([
        torch.full_like(x, 1 / math.sqrt(4 * math.pi)), -a1 * y, a1 * z, -a1 * x,
        a2 * x * y, -a2 * y * z, a20 * (2 * zz - xx - yy), -a2 * x * z, a22 * (xx - yy),
        -a33 * y * (3 * xx - yy), a32 * x * y * z, -a31 * y * (4 * zz - xx - yy),
        a30 * z * (2 * zz - 3 * xx - 3 * yy), -a31 * x * (4 * zz - xx - yy), a34 * z * (xx - yy),
        -a33 * x * (xx - 3 * yy)], 1)


def _project64(sc, cam, tile):
    """Depth, 2D mean, conic (a, b, c), colour and tile rect (x0, y0, x1, y1) of every Gaussian; empty rect: culled."""
    W = torch.from_numpy(np.asarray(cam.viewmat, np.float64)).cuda()
    m, s, q, o = sc.means.double(), sc.scales.double(), sc.quats.double(), sc.opacities.double()
    R, t = W[:3, :3], W[:3, 3]
    xc, yc, zc = (m @ R.T + t).unbind(1)
    vis = (zc > cam.near) & (zc < cam.far) & (o >= 1 / 255)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    Rq = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                      2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                      2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = R @ (Rq * s[:, None, :])
    S = M @ M.transpose(1, 2)
    lim = lambda v, c, size, f: torch.clamp(v, -1.3 * c / f, 1.3 * (size - c) / f)  # noqa: E731
    u, v = lim(xc / zc, cam.cx, cam.width, cam.fx), lim(yc / zc, cam.cy, cam.height, cam.fy)
    z0 = torch.zeros_like(zc)
    J = torch.stack([cam.fx / zc, z0, -cam.fx * u / zc, z0, cam.fy / zc, -cam.fy * v / zc], 1).view(-1, 2, 3)
    C2 = J @ S @ J.transpose(1, 2)
    a, b, c = C2[:, 0, 0] + 0.3, C2[:, 0, 1], C2[:, 1, 1] + 0.3
    det = a * c - b * b
    vis &= det > 0
    px, py = cam.fx * xc / zc + cam.cx, cam.fy * yc / zc + cam.cy
    mid = 0.5 * (a + c)
    r = torch.ceil(3 * torch.sqrt(mid + torch.sqrt(torch.clamp(mid * mid - det, min=0.01))))
    tx, ty = -(-cam.width // tile), -(-cam.height // tile)
    rect = torch.stack([torch.floor((px - r) / tile).clamp(0, tx), torch.floor((py - r) / tile).clamp(0, ty),
                        torch.ceil((px + r) / tile).clamp(0, tx), torch.ceil((py + r) / tile).clamp(0, ty)], 1)
    rect = torch.where(vis[:, None], rect, torch.zeros_like(rect)).long()
    d = m + R.T @ t
    Y = _sh_basis(d / d.norm(dim=1, keepdim=True))[:, :sc.sh.shape[1]]
    col = torch.clamp((Y[:, :, None] * sc.sh.double()).sum(1) + 0.5, min=0)
    return zc, torch.stack([px, py], 1), torch.stack([c / det, -b / det, a / det], 1), col, rect


def _lists64(z, rect, cam, tile):
    """Per-tile lists in (depth, id) order: offsets [T + 1] and Gaussian ids."""
    tx, ty = -(-cam.width // tile), -(-cam.height // tile)
    wh = (rect[:, 2:] - rect[:, :2]).clamp(min=0)
    cnt = wh[:, 0] * wh[:, 1]
    order = torch.argsort(z.float(), stable=True)
    cnt = cnt[order]
    rank = torch.repeat_interleave(torch.arange(cnt.numel(), device="cuda"), cnt)
    first = torch.cumsum(cnt, 0) - cnt
    k = torch.arange(rank.numel(), device="cuda") - first[rank]
    ro, wo = rect[order], wh[order, 0].clamp(min=1)
    t = (ro[rank, 1] + k // wo[rank]) * tx + ro[rank, 0] + k % wo[rank]
    del k
    t, at = torch.sort(t.int(), stable=True)
    off = torch.searchsorted(t, torch.arange(tx * ty + 1, device="cuda", dtype=torch.int32))
    return off, order[rank[at]]


def _composite64(o, mean, conic, col, off, gids, cam, tile, up=None):
    """rgb, alpha and, given upstream gradients, the gradient fields; chunks of
    each tile's list front to back until every pixel of the tile has stopped."""
    tx, H, W, n = -(-cam.width // tile), cam.height, cam.width, o.numel()
    T_all = off.numel() - 1
    P = tile * tile
    bg = torch.tensor(np.float32(_BG), dtype=torch.float64, device="cuda")
    img = torch.zeros(H * W, 3, dtype=torch.float64, device="cuda")
    trans = torch.ones(H * W, dtype=torch.float64, device="cuda")
    grads = torch.zeros(n, 9, dtype=torch.float64, device="cuda") if up is not None else None
    tb, Lc = max(1, (3 << 19) // P), 48
    for t0 in range(0, T_all, tb):
        tid = torch.arange(t0, min(T_all, t0 + tb), device="cuda")
        lx = torch.arange(P, device="cuda") % tile
        ly = torch.arange(P, device="cuda") // tile
        gx, gy = (tid % tx)[:, None] * tile + lx, (tid // tx)[:, None] * tile + ly
        inside = (gx < W) & (gy < H)
        pix = (gy * W + gx)[inside]

        def sweep(back):
            act = torch.arange(tid.numel(), device="cuda")
            T = torch.ones(tid.numel(), P, dtype=torch.float64, device="cuda")
            C = torch.zeros(tid.numel(), P, 3, dtype=torch.float64, device="cuda")
            done = ~inside
            pos = off[tid].clone()
            while act.numel():
                idx = pos[act][:, None] + torch.arange(Lc, device="cuda")
                live = idx < off[tid[act] + 1][:, None]
                g = gids[idx.clamp(max=gids.numel() - 1)]
                dx = mean[g, 0][:, :, None] - (gx[act][:, None] + 0.5)
                dy = mean[g, 1][:, :, None] - (gy[act][:, None] + 0.5)
                cn = conic[g]
                q = 0.5 * (cn[..., 0:1] * dx * dx + cn[..., 2:3] * dy * dy) + cn[..., 1:2] * dx * dy
                e = torch.exp(-q)
                oe = o[g][:, :, None] * e
                al = torch.clamp(oe, max=0.99)
                ok = live[:, :, None] & (q >= 0) & (al >= 1 / 255) & ~done[act][:, None]
                al = torch.where(ok, al, 0.0)
                Tn = T[act][:, None] * torch.cumprod(1 - al, 1)
                ok &= Tn >= 1e-4
                Ti = Tn / (1 - al)
                w = torch.where(ok, al * Ti, 0.0)
                if back is not None:
                    Gc, GT, GTot = back  # dL/drgb, T_N dL/dalpha, dL/drgb . (final colour with background)
                    gc = torch.einsum("tpc,tlc->tlp", Gc[act], col[g])
                    behind = GTot[act][:, None] - torch.einsum("tpc,tpc->tp", Gc[act], C[act])[:, None] - torch.cumsum(gc * w, 1)
                    dl = gc * Ti - (behind - GT[act][:, None]) / (1 - al)
                    v = torch.where(ok & (oe <= 0.99), dl * e, 0.0)
                    og = -o[g][:, :, None] * v
                    part = torch.stack([(og * (cn[..., 0:1] * dx + cn[..., 1:2] * dy)).sum(2),
                                        (og * (cn[..., 1:2] * dx + cn[..., 2:3] * dy)).sum(2),
                                        0.5 * (og * dx * dx).sum(2), (og * dx * dy).sum(2), 0.5 * (og * dy * dy).sum(2),
                                        v.sum(2)], 2)
                    part = torch.cat([part, torch.einsum("tlp,tpc->tlc", w, Gc[act])], 2)
                    grads.index_add_(0, g[live], part[live])
                C[act] += torch.einsum("tlp,tlc->tpc", w, col[g])
                stop = Tn[:, -1] < 1e-4
                low = torch.where(ok, Tn, 2.0).amin(1)  # the last applied entry's
                T[act] = torch.where(done[act] | (low > 1.5), T[act], low)
                done[act] |= stop
                pos[act] += Lc
                act = act[(pos[act] < off[tid[act] + 1]) & ~done[act].all(1)]
            return C, T

        C, T = sweep(None)
        full = C + T[..., None] * bg
        img[pix], trans[pix] = full[inside], T[inside]
        if up is not None:
            Gc = torch.zeros_like(C)
            Gc[inside] = up[0].double().view(-1, 3)[pix]
            dA = torch.zeros_like(T)
            dA[inside] = up[1].double().view(-1)[pix]
            sweep((Gc, T * dA, (Gc * full).sum(2)))
    out = [img.view(H, W, 3), (1 - trans).view(H, W)]
    if up is not None:
        z1, z2 = torch.zeros_like(grads[:, :1]), torch.zeros_like(grads[:, :2])
        out += [grads[:, 0:4].contiguous(), torch.cat([grads[:, 4:6], z2], 1), torch.cat([grads[:, 6:9], z1], 1)]
    return out


def _fit64(case, seed):
    X, y, P = (t.double() if t.is_floating_point() else t.long() for t in _fit_inputs(case, seed))
    F, H, C = G.PLAN_FEATURES, G.PLAN_HIDDEN, G.PLAN_CLASSES
    P.requires_grad_()
    W1, b1, W2, b2, W3, b3 = torch.split(P, [H * F, H, H * H, H, C * H, C])
    h = torch.relu(X @ W1.view(H, F).T + b1)
    h = torch.relu(h @ W2.view(H, H).T + b2)
    logits = h @ W3.view(C, H).T + b3
    loss = torch.nn.functional.cross_entropy(logits, y)
    (g,) = torch.autograd.grad(loss, P)
    b1_, b2_, lr, eps = (float(np.float32(v)) for v in (0.9, 0.999, 3e-3, 1e-8))
    m, v = (1 - b1_) * g, (1 - b2_) * g * g
    new = P.detach() - lr * (m / (1 - b1_)) / (torch.sqrt(v / (1 - b2_)) + eps)
    return [loss.detach().view(1), logits.detach(), g, new, m, v]


def exact(case, seed):
    if case["path"] == "fit":
        return _fit64(case, seed)
    if case["mode"] == "paper":
        return None  # approximate by definition, and its order inside a bin is open
    sc, centres = _scene(case, seed)
    res = []
    for cam in _cameras(case, seed, centres):
        z, mean, conic, col, rect = _project64(sc, cam, case["tile"])
        off, gids = _lists64(z, rect, cam, case["tile"])
        up = _upstream(cam, seed) if case["path"] in ("train", "stages") else None
        res.append(_composite64(sc.opacities.double(), mean, conic, col, off, gids, cam, case["tile"], up))
        del off, gids
    if case["path"] == "batch":
        return [(r[0], r[1], None) for r in res]
    r = res[0]
    if case["path"] == "stages":
        return r
    return [r[0], r[1], None] + r[2:]  # the last id follows float32 rounding
