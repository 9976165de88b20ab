"""Timed cases of the library: the calls a user's program makes, over the sizes it makes them at.

A case is a dict of plain values; ``kind`` names the call:

* ``bounds``  -- ``Bounds.compute``: Alg. 1's interval, count and offsets of every ray;
* ``fuse``    -- ``Grid.init``, ``Grid.integrate`` and ``Grid.inside_mask``: depth maps into a volume;
* ``raycast`` -- ``Grid.init`` and ``Grid.integrate_raycast``: the ray-casting form of the fusion;
* ``render``  -- ``Renderer.render`` over bounds in hand;
* ``view``    -- ``Bounds.compute`` and ``Renderer.render``: one whole novel view;
* ``hier``    -- ``HierRenderer.render``: the coarse + fine comparator over the whole ray;
* ``train``   -- ``RenderFunction``, an L1 colour + eikonal loss, and its backward.

Scenes, camera models, parameters and networks are those of ``synth``: the unit sphere with the
tiny networks and the 8 x 6 x 3 m room with the room networks.  The seed chooses camera poses,
depth noise, ray subsets and colour targets.  Grids are fused from seeded depth maps.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_17878_gb300 import synth
from paper_2311_17878_gb300 import tsdfs as T

DEV = "cuda"
PREC = {"f32": T.TSDFS_PREC_F32, "f16": T.TSDFS_PREC_F16, "bf16": T.TSDFS_PREC_BF16, "bf16x2": T.TSDFS_PREC_BF16X2}
OPACITY = {"neus": 0, "volsdf": 1}
# mean samples of a ray inside its bound (room: 2-voxel spacing; sphere: 1-voxel spacing, most rays miss)
SAMPLES_PER_RAY = {"room": 14.0, "sphere": 23.0}
# algorithmic flops of one sample: SDF forward, reverse-mode gradient, colour (room / tiny networks)
FLOPS_PER_SAMPLE = {"room": 2.25e6, "sphere": 6.2e4}
SDF_FLOPS = {"room": 0.92e6, "sphere": 1.9e4}
PARAMS = {"room": 745_000, "sphere": 15_600}


def listed():
    return [
        # a few hundred rays probed against a small object's volume: a pick or a collision test
        dict(name="bounds_rays", kind="bounds", scene="sphere", n=64, w=25, h=20, mask=False, dtype="f32"),
        # one 640 x 480 novel view of the room against its 256^3 volume
        dict(name="bounds_view", kind="bounds", scene="room", n=256, w=640, h=480, mask=True, dtype="f32"),
        # the room's whole capture, 100 depth maps of 640 x 480, into a fresh 256^3 volume
        dict(name="fuse_scene", kind="fuse", scene="room", n=256, nx=256, ny=256, nz=256, views=100, w=640, h=480,
             dtype="f32", radius=2),
        # a few new frames into a half-precision volume whose sides are no multiples of anything
        dict(name="fuse_frames", kind="fuse", scene="room", n=300, nx=300, ny=225, nz=121, views=3, w=320, h=240,
             dtype="f16", radius=2),
        # the printed form of the fusion, every pixel's ray walked
        dict(name="raycast_scene", kind="raycast", scene="room", n=256, nx=256, ny=256, nz=256, views=10, w=640, h=480,
             dtype="f32"),
        # a whole novel view with half-precision networks: the headline use
        dict(name="view_f16", kind="view", scene="room", n=256, w=640, h=480, prec="f16", opacity="neus"),
        # a thumbnail or a tile of a progressive viewer
        dict(name="chunk_f16", kind="render", scene="room", n=256, w=37, h=31, prec="f16", opacity="neus"),
        # a chunk of an image with single-precision networks, the library's default precision
        dict(name="chunk_f32", kind="render", scene="room", n=256, w=101, h=81, prec="f32", opacity="neus"),
        # the small object with its small networks in single precision
        dict(name="tiny_f32", kind="render", scene="sphere", n=64, w=64, h=64, prec="f32", opacity="neus"),
        # a preview image with split-operand networks and the density form of the opacity
        dict(name="chunk_split", kind="render", scene="room", n=256, w=160, h=120, prec="bf16x2", opacity="volsdf"),
        # the 64 + 32 sampler over a preview image
        dict(name="hier_f16", kind="hier", scene="room", n=256, w=80, h=60, prec="f16", coarse=64, fine=32),
        # a training step over a batch of random rays of the captured views
        dict(name="train_step", kind="train", scene="room", n=256, rays=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bounds", "fuse", "raycast", "view", "render", "render", "render", "hier", "train"])
    if kind in ("fuse", "raycast"):
        n = _log_int(rng, 48, 256)
        side = [max(16, int(n * rng.uniform(0.4, 1.0))) for _ in range(3)]
        most = 100 if kind == "fuse" else 10
        w = _log_int(rng, 64, 640)
        c = dict(kind=kind, scene="room", n=n, nx=side[0], ny=side[1], nz=side[2], views=_log_int(rng, 1, most), w=w,
                 h=max(16, int(w * 0.75)), dtype=rng.choice(["f32", "f16"]))
        return dict(c, radius=rng.choice([1, 2, 3])) if kind == "fuse" else c
    if kind == "train":
        return dict(kind=kind, scene="room", n=rng.choice([128, 192, 256]), rays=_log_int(rng, 256, 8000))
    scene = rng.choice(["room", "room", "sphere"])
    n = rng.choice([128, 192, 256]) if scene == "room" else rng.choice([48, 64, 96])
    # sides of the image: the largest call of each kind costs no more than the listed one
    prec = rng.choice(["f16", "f32", "bf16x2", "bf16"]) if kind != "view" else rng.choice(["f16", "bf16x2"])
    most = {"bounds": 620, "view": 400 if prec == "f16" else 240, "hier": 80 if prec != "f32" else 32,
            "render": 90 if prec == "f32" else 200}[kind]
    w = _log_int(rng, 16, most)
    c = dict(kind=kind, scene=scene, n=n, w=w, h=max(8, int(w * rng.uniform(0.6, 0.8))))
    if kind == "bounds":
        return dict(c, mask=rng.random() < 0.7, dtype=rng.choice(["f32", "f16"]))
    c["prec"] = prec
    if kind == "hier":
        return dict(c, coarse=rng.choice([64, 8, 33]), fine=rng.choice([32, 4, 17]))
    return dict(c, opacity=rng.choice(["neus", "neus", "volsdf"]))


# ---- inputs ------------------------------------------------------------------------------
def _scene(case):
    return synth.SphereScene() if case["scene"] == "sphere" else synth.room_scene()


def _grid_spec(case, dtype="f32", box=None):
    """The scene's grid at ``n`` voxels a side; ``box``: a part of it of so many voxels, about its centre."""
    n = case["n"]
    if case["scene"] == "sphere":
        vs = 1.0 / n
        spec = synth.GridSpec(n, n, n, (-0.5, -0.5, -0.5), vs, 3 * vs, dtype)
    else:
        g = synth.room_grid(n)
        spec = synth.GridSpec(n, n, n, g.origin, g.voxel_size, g.trunc, dtype)
    if box is not None:
        vs, side = spec.voxel_size, n * spec.voxel_size
        # centred on the whole grid
        origin = tuple(o + 0.5 * (side - b * vs) for o, b in zip(spec.origin, box))
        spec = synth.GridSpec(box[0], box[1], box[2], origin, vs, spec.trunc, dtype)
    return spec


def _params(case, spec):
    vs = spec.voxel_size
    if case["scene"] == "sphere":
        return synth.BoundsParams(d_s=vs, t_near=0.0, t_far=4.0, step=vs, n_max=32)
    return synth.BoundsParams(d_s=vs, t_near=0.05, t_far=12.0, step=2 * vs, n_max=64)


def _poses(case, rng, n):
    if case["scene"] == "sphere":
        out = []
        for _ in range(n):
            az, el = rng.uniform(0, 2 * np.pi), rng.uniform(-0.5, 0.5)
            eye = 2.0 * np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
            out.append(synth.look_at(eye, (0, 0, 0)))
        return np.array(out)
    return synth.sample_free_poses(_scene(case), rng, n)


def _focal(case, w):
    return float(w) if case["scene"] == "sphere" else 500.0 * w / 640.0


def _capture(case, rng, gen, views, w, h):
    """Seeded depth maps (range along the pixel's ray, 5 mm noise in the room) with K and c2w."""
    poses, f, scene = _poses(case, rng, views), _focal(case, w), _scene(case)
    if case["scene"] == "sphere":
        depth = synth.render_depth_maps_torch(scene, poses, f, f, w / 2.0, h / 2.0, w, h, device=DEV)
    else:
        depth = synth.render_depth_maps_torch_f32(scene, poses, f, f, w / 2.0, h / 2.0, w, h, device=DEV)
        depth += 0.005 * torch.randn(depth.shape, generator=gen, device=DEV)
    K = torch.tensor([f, f, w / 2.0, h / 2.0], dtype=torch.float32, device=DEV).repeat(views, 1)
    c2w = torch.tensor(poses.reshape(views, 12), dtype=torch.float32, device=DEV)
    return depth.contiguous(), K, c2w


def _fused(case, rng, gen, dtype="f32"):
    spec = _grid_spec(case, dtype)
    views = 12 if case["scene"] == "sphere" else 40
    return T.Grid(spec).init().integrate(*_capture(case, rng, gen, views, 160 if case["scene"] == "sphere" else 320,
                                                   160 if case["scene"] == "sphere" else 240))


def _rays(case, rng):
    f = _focal(case, case["w"])
    o, d = synth.pinhole_rays(_poses(case, rng, 1)[0], f, f, case["w"] / 2.0, case["h"] / 2.0, case["w"], case["h"])
    return torch.tensor(o, dtype=torch.float32, device=DEV), torch.tensor(d, dtype=torch.float32, device=DEV)


def _spec(case):
    spec = synth.scene_mlp("tiny" if case["scene"] == "sphere" else "room")
    spec.opacity = OPACITY[case.get("opacity", "neus")]
    return spec


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    kind = case["kind"]
    s = {"kind": kind}
    if kind in ("fuse", "raycast"):
        s["depth"], s["K"], s["c2w"] = _capture(case, rng, gen, case["views"], case["w"], case["h"])
        s["grid"] = T.Grid(_grid_spec(case, case["dtype"], (case["nx"], case["ny"], case["nz"])))
        s["radius"] = case.get("radius", 0)
        if kind == "raycast":
            s["ws"] = torch.empty(T.tsdfs_raycast_workspace_size(s["grid"]), dtype=torch.uint8, device=DEV)
        return s
    grid = s["grid"] = _fused(case, rng, gen, case.get("dtype", "f32"))
    bp = _params(case, grid.spec)
    s["bp"] = T.bounds_params(bp)
    s["mask"] = grid.inside_mask(bp.nb_radius) if case.get("mask", True) else None
    if kind == "train":
        n = case["rays"]
        poses = _poses(case, rng, 64)
        views = synth.Views(np.tile(np.array([500.0, 500.0, 320.0, 240.0], np.float32), (64, 1)),
                            poses.reshape(64, 12).astype(np.float32), None, 640, 480)
        o, d, _, _, _ = synth.random_rays_from_views(views, n, seed=int(seed))
        s["o"], s["d"] = torch.tensor(o, device=DEV), torch.tensor(d, device=DEV)
        s["target"] = torch.rand((n, 3), device=DEV, generator=gen)
    else:
        s["o"], s["d"] = _rays(case, rng)
    n = s["o"].shape[0]
    if kind == "hier":
        s["mlp"] = T.Mlp(_spec(case), PREC[case["prec"]])
        s["renderer"] = T.HierRenderer(s["mlp"], n, n_coarse=case["coarse"], n_fine=case["fine"])
        return s
    s["bounds"] = T.Bounds(n)
    if kind == "bounds":
        return s
    cap = n * max(bp.n_max, bp.n_fallback)
    s["mlp"] = T.Mlp(_spec(case), PREC[case.get("prec", "f32")])
    if kind == "view":
        s["renderer"] = T.Renderer(s["mlp"], n, cap)
        return s
    s["bounds"].compute(grid, s["o"], s["d"], s["bp"], s["mask"])
    if kind == "render":
        s["renderer"] = T.Renderer(s["mlp"], n, cap)
        return s
    s["cap"] = cap
    s["n_bounded"] = torch.clamp((s["bounds"].n * (s["bounds"].status == T.TSDFS_BOUNDED)).sum(), min=1)
    s["sdf_w"] = s["mlp"].sdf_w.clone().requires_grad_(True)
    s["rgb_w"] = s["mlp"].rgb_w.clone().requires_grad_(True)
    return s


# ---- one pass ------------------------------------------------------------------------------
def _bounds_out(b):
    return {"t_n": b.t_n, "t_f": b.t_f, "n": b.n, "offsets": b.offsets, "t_zero": b.t_zero, "status": b.status}


def _render_out(o, eik=True):
    out = {"rgb": o.rgb, "depth": o.depth, "wsum": o.wsum, "normal": o.normal}
    return dict(out, eik=o.eik) if eik else out


def run(s):
    kind, grid = s["kind"], s["grid"]
    if kind == "fuse":
        grid.init().integrate(s["depth"], s["K"], s["c2w"])
        return {"V": grid.V, "W": grid.W, "mask": grid.inside_mask(s["radius"])}
    if kind == "raycast":
        grid.init().integrate_raycast(s["depth"], s["K"], s["c2w"], s["ws"])
        return {"V": grid.V, "W": grid.W}
    if kind == "bounds":
        return _bounds_out(s["bounds"].compute(grid, s["o"], s["d"], s["bp"], s["mask"]))
    if kind == "render":
        return _render_out(s["renderer"].render(s["o"], s["d"], s["bounds"]))
    if kind == "view":
        b = s["bounds"].compute(grid, s["o"], s["d"], s["bp"], s["mask"])
        return dict(_render_out(s["renderer"].render(s["o"], s["d"], b)), n=b.n, status=b.status)
    if kind == "hier":
        return _render_out(s["renderer"].render(grid, s["o"], s["d"], s["bp"].t_near, s["bp"].t_far), eik=False)
    sdf_w, rgb_w = s["sdf_w"], s["rgb_w"]
    sdf_w.grad = rgb_w.grad = None
    rgb, depth, eik = T.RenderFunction.apply(sdf_w, rgb_w, s["mlp"], s["o"], s["d"], s["bounds"], s["cap"])
    loss = (rgb - s["target"]).abs().mean() + 0.1 * eik.sum() / s["n_bounded"]
    loss.backward()
    return {"loss": loss.detach(), "rgb": rgb.detach(), "depth": depth.detach(), "d_sdf": sdf_w.grad, "d_rgb": rgb_w.grad}


def work(case):
    kind = case["kind"]
    if kind in ("fuse", "raycast"):
        vox, pix = case["nx"] * case["ny"] * case["nz"], case["views"] * case["w"] * case["h"]
        # volume written (and its mask), maps read; a projection and an update per voxel and view that sees it
        # (about one in four), or per voxel that a pixel's ray crosses
        per = 3 if case["dtype"] == "f16" else 5
        upd = 0.25 * vox * case["views"] if kind == "fuse" else 0.25 * case["n"] * pix
        return {"bytes": vox * (per + (1 / 8 if kind == "fuse" else 0)) + 4.0 * pix, "flops": 40.0 * upd}
    rays = case["rays"] if kind == "train" else case["w"] * case["h"]
    scene = case["scene"]
    if kind == "bounds":
        vox = 0.5 * case["n"]
        return {"bytes": 24.0 * rays + 21.0 * rays + 4.0 * rays * vox, "flops": 30.0 * rays * vox}
    par = PARAMS[scene]
    if kind == "hier":
        c, f = case["coarse"], case["fine"]
        return {"bytes": 56.0 * rays + 4.0 * par,
                "flops": rays * (c * SDF_FLOPS[scene] + (c + f) * FLOPS_PER_SAMPLE[scene])}
    ns = rays * SAMPLES_PER_RAY[scene]
    if kind == "train":
        # forward, then twice that for the adjoints of activations and parameters
        return {"bytes": 80.0 * rays + 8.0 * par, "flops": 3.0 * ns * FLOPS_PER_SAMPLE[scene]}
    return {"bytes": 80.0 * rays + (2.0 if case["prec"] != "f32" else 4.0) * par + (4.0 * rays * case["n"] / 2 if kind == "view" else 0.0),
            "flops": ns * FLOPS_PER_SAMPLE[scene]}


# ---- the same in 64 bits ---------------------------------------------------------------------
D64 = torch.float64


def _geometry(grid):
    c = grid.c
    return [c.nx, c.ny, c.nz], [float(v) for v in c.origin], float(c.voxel_size), float(c.trunc)


def _clip64(o, d, dims, org, vs, t_near, t_far):
    lo = torch.tensor(org, dtype=D64, device=DEV)
    hi = lo + vs * torch.tensor(dims, dtype=D64, device=DEV)
    t1, t2 = (lo - o) / d, (hi - o) / d
    zero = d == 0
    out = (zero & ((o < lo) | (o > hi))).any(1)
    inf = torch.full_like(t1, float("inf"))
    t0 = torch.clamp(torch.where(zero, -inf, torch.minimum(t1, t2)).amax(1), min=t_near)
    te = torch.clamp(torch.where(zero, inf, torch.maximum(t1, t2)).amin(1), max=t_far)
    return t0, te, ~out & (t0 < te)


def _walk64(o, d, t0, dims, org, vs):
    """Voxel walk of many rays: returns the start voxel and a step function (X, t) -> (X, t, in grid)."""
    lo, n = torch.tensor(org, dtype=D64, device=DEV), torch.tensor(dims, device=DEV)
    X = torch.minimum(torch.clamp(torch.floor((o + t0[:, None] * d - lo) / vs), min=0).long(), n - 1)
    step = torch.sign(d).long()

    def nxt(X):
        t = torch.where(step != 0, (lo + (X + (step > 0)) * vs - o) / d, torch.full_like(d, float("inf")))
        tm, a = t.min(1)
        X = X + torch.nn.functional.one_hot(a, 3) * step
        return X, tm, ((X >= 0) & (X < n)).all(1)

    return X, nxt


def _bounds64(s, case):
    dims, org, vs, trunc = _geometry(s["grid"])
    bp = s["bp"]
    o, d = s["o"].to(D64), s["d"].to(D64)
    V = s["grid"].V.to(D64)
    r = bp.nb_radius
    pad = torch.nn.functional.pad(V[None, None], (r,) * 6, value=-1.0)
    inside = (torch.nn.functional.max_pool3d(pad, 2 * r + 1, stride=1)[0, 0] < 0)
    t0, te, hit = _clip64(o, d, dims, org, vs, bp.t_near, bp.t_far)
    t0, te = torch.where(hit, t0, torch.zeros_like(t0)), torch.where(hit, te, torch.zeros_like(te))
    X, nxt = _walk64(o, d, t0, dims, org, vs)
    t, near, far = t0.clone(), hit.clone(), torch.zeros_like(hit)
    tn, tf, m = t0.clone(), te.clone(), torch.zeros_like(X[:, 0])
    for k in range(sum(dims) + 8):
        if k % 16 == 0 and not bool((near | far).any()):
            break
        Xc = torch.minimum(torch.clamp(X, min=0), torch.tensor(dims, device=DEV) - 1)
        at = (Xc[:, 2], Xc[:, 1], Xc[:, 0])
        found = near & (V[at] <= bp.d_s / trunc)
        tn = torch.where(found, t, tn)
        near, far = near & ~found, far | found
        m = torch.where(inside[at], m + 1, torch.zeros_like(m)) * far
        X, t, ok = nxt(X)
        tc = torch.minimum(t, te)
        end = far & (m == bp.m_confirm)
        tf = torch.where(end, tc, tf)
        live = ok & (t < te)
        near, far = near & live, far & ~end & live
    return {"t_n": tn, "t_f": tf, "n": None, "offsets": None, "t_zero": None, "status": None}


def _fuse64(s, case):
    dims, org, vs, trunc = _geometry(s["grid"])
    nx, ny, nz = dims
    z, y, x = torch.meshgrid(*[(torch.arange(k, device=DEV, dtype=D64) + 0.5) * vs + org[a]
                               for a, k in ((2, nz), (1, ny), (0, nx))], indexing="ij")
    V, W = torch.full((nz, ny, nx), -1.0, dtype=D64, device=DEV), torch.zeros((nz, ny, nx), dtype=D64, device=DEV)
    _, H, Wd = s["depth"].shape
    for v in range(s["depth"].shape[0]):
        P = s["c2w"][v].to(D64).reshape(3, 4).tolist()
        fx, fy, cx, cy = s["K"][v].to(D64).tolist()
        dx, dy, dz = x - P[0][3], y - P[1][3], z - P[2][3]
        xc, yc, zc = (P[0][k] * dx + P[1][k] * dy + P[2][k] * dz for k in range(3))
        u, w = fx * (xc / zc) + cx, fy * (yc / zc) + cy
        at = torch.nonzero(((zc > 0) & (u >= 0) & (u < Wd) & (w >= 0) & (w < H)).reshape(-1))[:, 0]
        px, py = u.reshape(-1)[at].long(), w.reshape(-1)[at].long()
        D = s["depth"][v].to(D64)[py, px]
        a, b = (px + 0.5 - cx) / fx, (py + 0.5 - cy) / fy
        proj = (a * xc.reshape(-1)[at] + b * yc.reshape(-1)[at] + zc.reshape(-1)[at]) / torch.sqrt(a * a + b * b + 1)
        sd = torch.clamp(D - proj, -trunc, trunc)
        keep = sd > -trunc
        at, sd = at[keep], sd[keep] / trunc
        Vf, Wf = V.view(-1), W.view(-1)
        Vf[at] = (Wf[at] * Vf[at] + sd) / (Wf[at] + 1)
        Wf[at] = torch.clamp(Wf[at] + 1, max=255)
    return {"V": V, "W": None, "mask": None}


def _raycast64(s, case):
    dims, org, vs, trunc = _geometry(s["grid"])
    nx, ny, nz = dims
    V, W = torch.full((nz * ny * nx,), -1.0, dtype=D64, device=DEV), torch.zeros(nz * ny * nx, dtype=D64, device=DEV)
    _, H, Wd = s["depth"].shape
    lo = torch.tensor(org, dtype=D64, device=DEV)
    for v in range(s["depth"].shape[0]):
        P = s["c2w"][v].to(D64).reshape(3, 4)
        fx, fy, cx, cy = s["K"][v].to(D64).tolist()
        py, px = torch.meshgrid(torch.arange(H, device=DEV, dtype=D64), torch.arange(Wd, device=DEV, dtype=D64), indexing="ij")
        dc = torch.stack([(px + 0.5 - cx) / fx, (py + 0.5 - cy) / fy, torch.ones_like(px)], -1).reshape(-1, 3)
        d = dc @ P[:, :3].T
        d = d / torch.linalg.norm(d, dim=1, keepdim=True)
        o = P[:, 3].expand_as(d).contiguous()
        D = s["depth"][v].to(D64).reshape(-1)
        t, te, live = _clip64(o, d, dims, org, vs, 0.0, float("inf"))
        t = torch.where(live, t, torch.zeros_like(t))
        X, nxt = _walk64(o, d, t, dims, org, vs)
        p, add, cnt = o + D[:, None] * d, torch.zeros_like(V), torch.zeros_like(V)
        for k in range(sum(dims) + 8):
            if k % 16 == 0 and not bool(live.any()):
                break
            e = ((p - (lo + (X + 0.5) * vs)) * d).sum(1)
            sd = torch.where(torch.isinf(D), torch.full_like(D, trunc), torch.clamp(e, -trunc, trunc))
            live = live & (t < te) & (sd > -trunc)
            Xc = torch.minimum(torch.clamp(X, min=0), torch.tensor(dims, device=DEV) - 1)
            at = (Xc[:, 2] * ny + Xc[:, 1]) * nx + Xc[:, 0]
            add.index_add_(0, at[live], sd[live] / trunc)
            cnt.index_add_(0, at[live], torch.ones_like(sd[live]))
            X, t, ok = nxt(X)
            live = live & ok
        V = torch.where(cnt > 0, (W * V + add) / torch.clamp(W + cnt, min=1), V)
        W = torch.clamp(W + cnt, max=255)
    return {"V": V.view(nz, ny, nx), "W": None}


def _net64(spec, sdf_w=None, rgb_w=None):
    """Layers (W, b) of both networks in 64 bits, from the packed parameters where they are given."""
    def layers(ws, packed):
        out, k = [], 0
        for W, b in ws:
            if packed is None:
                out.append((torch.tensor(np.asarray(W), dtype=D64, device=DEV), torch.tensor(np.asarray(b), dtype=D64, device=DEV)))
            else:
                out.append((packed[k:k + W.size].reshape(W.shape), packed[k + W.size:k + W.size + b.size]))
                k += W.size + b.size
        return out
    return layers(spec.sdf, sdf_w), layers(spec.rgb, rgb_w)


def _encode64(x, octaves):
    parts, jac = [x], [torch.eye(3, dtype=D64, device=DEV).expand(x.shape[0], 3, 3)]
    for k in range(octaves):
        f = 2.0 ** k
        parts += [torch.sin(f * x), torch.cos(f * x)]
        jac += [torch.diag_embed(f * torch.cos(f * x)), torch.diag_embed(-f * torch.sin(f * x))]
    return torch.cat(parts, 1), torch.cat(jac, 2)


def _sdf64(spec, net, x, grad=True):
    xt = (x - torch.tensor(spec.center, dtype=torch.float32, device=DEV).to(D64)) / float(np.float32(spec.scale))
    g, jg = _encode64(xt, spec.pe_sdf)
    h, dh = g, jg
    for l, (W, b) in enumerate(net[0]):
        if l == spec.skip_layer:
            h, dh = torch.cat([h, g], 1) / math.sqrt(2.0), torch.cat([dh, jg], 2) / math.sqrt(2.0)
        z = h @ W.T + b
        dz = dh @ W.T if grad else dh
        if l + 1 < len(net[0]):
            bz = spec.beta * z
            h = torch.where(bz > 20, z, torch.log1p(torch.exp(torch.clamp(bz, max=20.0))) / spec.beta)
            dh = torch.where(bz > 20, torch.ones_like(z), torch.sigmoid(bz))[:, None] * dz if grad else dh
        else:
            h, dh = z, dz
    return xt, spec.scale * h[:, 0], dh[:, :, 0] if grad else None, h[:, 1:]


def _samples64(spec, net, o, d, t):
    """f, v . grad f, colour, unit normal and |grad f| at points o + t d."""
    xt, f, g, feat = _sdf64(spec, net, o + t[:, None] * d)
    gn = torch.linalg.norm(g, dim=1)
    nh = g / gn[:, None]
    h = torch.cat([xt, _encode64(d, spec.pe_dir)[0], nh, feat], 1)
    for l, (W, b) in enumerate(net[1]):
        z = h @ W.T + b
        h = torch.relu(z) if l + 1 < len(net[1]) else torch.sigmoid(z)
    return f, (g * d).sum(1), h, nh, gn


def _alpha64(spec, f, dd, dl):
    s, eps = float(np.float32(spec.inv_s)), float(np.float32(spec.alpha_eps))
    if spec.opacity == OPACITY["volsdf"]:
        e = 0.5 * torch.exp(-s * f.abs())
        return -torch.expm1(-s * torch.where(f >= 0, e, 1 - e) * dl)
    c = torch.clamp(dd, max=0.0)
    lo, hi = torch.sigmoid(s * (f - 0.5 * dl * c)), torch.sigmoid(s * (f + 0.5 * dl * c))
    return torch.clamp((lo - hi + eps) / (lo + eps), 0.0, 1.0)


def _composite64(spec, net, o, d, t, dl, cnt, bounded):
    """Rays' ragged samples t, dl (concatenated, cnt[r] of ray r) rendered; all in 64 bits."""
    R = o.shape[0]
    ray = torch.repeat_interleave(torch.arange(R, device=DEV), cnt)
    f, dd, rgb, nh, gn = _samples64(spec, net, o[ray], d[ray], t)
    al = _alpha64(spec, f, dd, dl)
    S = max(1, int(cnt.max())) if R else 1
    first = torch.cumsum(cnt, 0) - cnt
    col = torch.arange(t.shape[0], device=DEV) - first[ray]
    pad = torch.zeros((R, S), dtype=D64, device=DEV).index_put((ray, col), al)
    lt = torch.log1p(-torch.clamp(pad, max=1.0 - 2.0 ** -24))
    w = (torch.exp(torch.cumsum(lt, 1) - lt) * pad)[ray, col]
    tot = lambda v: torch.zeros((R,) + v.shape[1:], dtype=D64, device=DEV).index_add(0, ray, v)  # noqa: E731
    wsum = tot(w)
    ok = wsum >= 1e-8
    inv = torch.where(ok, 1 / torch.where(ok, wsum, torch.ones_like(wsum)), torch.zeros_like(wsum))
    return {"rgb": tot(w[:, None] * rgb), "depth": tot(w * t) * inv, "wsum": wsum, "normal": tot(w[:, None] * nh) * inv[:, None],
            "eik": tot((gn - 1) ** 2) * bounded}


def _ragged64(s, r0, r1):
    b = s["bounds"]
    cnt = b.n[r0:r1].long()
    ray = torch.repeat_interleave(torch.arange(r1 - r0, device=DEV), cnt)
    i = torch.arange(ray.shape[0], device=DEV) - (torch.cumsum(cnt, 0) - cnt)[ray]
    tn, tf = b.t_n[r0:r1].to(D64), b.t_f[r0:r1].to(D64)
    dl = ((tf - tn) / torch.clamp(cnt, min=1))[ray]
    return tn[ray] + (i + 0.5) * dl, dl, cnt, (b.status[r0:r1] == T.TSDFS_BOUNDED).to(D64)


def _hier64(s, case, spec, net, o, d):
    dims, org, vs, _ = _geometry(s["grid"])
    R, c, nf = o.shape[0], case["coarse"], case["fine"]
    t0, te, hit = _clip64(o, d, dims, org, vs, s["bp"].t_near, s["bp"].t_far)
    t0, te = torch.where(hit, t0, torch.zeros_like(t0)), torch.where(hit, te, torch.zeros_like(te))
    z = t0[:, None] + (torch.arange(c, device=DEV) + 0.5) * ((te - t0) / c)[:, None]
    f = _sdf64(spec, net, (o[:, None] + z[:, :, None] * d[:, None]).reshape(-1, 3), grad=False)[1].reshape(R, c)
    dz, mid = z[:, 1:] - z[:, :-1], 0.5 * (f[:, 1:] + f[:, :-1])
    slope = torch.where(dz > 0, (f[:, 1:] - f[:, :-1]) / dz, torch.zeros_like(dz))
    prev = torch.cat([torch.zeros_like(slope[:, :1]), slope[:, :-1]], 1)
    al = _alpha64(spec, mid, torch.clamp(torch.minimum(slope, prev), -1e3, 0.0), dz)
    w = al * torch.cumprod(torch.cat([torch.ones_like(al[:, :1]), 1 - al[:, :-1]], 1), 1) + 1e-5
    pdf = w / w.sum(1, keepdim=True)
    cdf = torch.cat([torch.zeros_like(pdf[:, :1]), torch.cumsum(pdf, 1)], 1)
    u = ((torch.arange(nf, device=DEV, dtype=D64) + 0.5) / nf).expand(R, nf).contiguous()
    j = torch.clamp(torch.searchsorted(cdf, u, right=True) - 1, 0, c - 2)
    zf = torch.gather(z, 1, j) + (u - torch.gather(cdf, 1, j)) / torch.gather(pdf, 1, j) * torch.gather(dz, 1, j)
    t = torch.sort(torch.cat([z, zf], 1), 1)[0]
    edge = torch.cat([t0[:, None], 0.5 * (t[:, 1:] + t[:, :-1]), te[:, None]], 1)
    dl = edge[:, 1:] - edge[:, :-1]
    cnt = torch.where(hit, c + nf, 0)
    return t[hit].reshape(-1), dl[hit].reshape(-1), cnt


def exact(case, seed):
    kind = case["kind"]
    s = prepare(case, seed)
    if kind in ("fuse", "raycast", "bounds"):
        return {"fuse": _fuse64, "raycast": _raycast64, "bounds": _bounds64}[kind](s, case)
    rays = s["o"].shape[0]
    per = {"hier": case.get("coarse", 0) + case.get("fine", 0)}.get(kind, SAMPLES_PER_RAY[case["scene"]])
    if kind == "view" or rays * per * FLOPS_PER_SAMPLE[case["scene"]] > 2e12:
        return None   # some 10^13 operations in 64 bits
    spec = _spec(case)
    o, d = s["o"].to(D64), s["d"].to(D64)
    per_chunk = max(64, int(60_000 / per))
    if kind == "train":
        wl = [s["sdf_w"].detach().to(D64).requires_grad_(True), s["rgb_w"].detach().to(D64).requires_grad_(True)]
        net, loss, outs = _net64(spec, *wl), 0.0, []
        target, nb = s["target"].to(D64), s["n_bounded"].to(D64)
        for r in range(0, rays, per_chunk):
            q = min(rays, r + per_chunk)
            t, dl, cnt, bounded = _ragged64(s, r, q)
            out = _composite64(spec, net, o[r:q], d[r:q], t, dl, cnt, bounded)
            part = (out["rgb"] - target[r:q]).abs().sum() / (3 * rays) + 0.1 * out["eik"].sum() / nb
            part.backward()
            loss = loss + part.detach()
            outs.append({k: out[k].detach() for k in ("rgb", "depth")})
        return {"loss": loss, "rgb": torch.cat([x["rgb"] for x in outs]), "depth": torch.cat([x["depth"] for x in outs]),
                "d_sdf": wl[0].grad, "d_rgb": wl[1].grad}
    net, outs = _net64(spec), []
    with torch.no_grad():
        for r in range(0, rays, per_chunk):
            q = min(rays, r + per_chunk)
            if kind == "hier":
                t, dl, cnt = _hier64(s, case, spec, net, o[r:q], d[r:q])
                bounded = torch.zeros(q - r, dtype=D64, device=DEV)
            else:
                t, dl, cnt, bounded = _ragged64(s, r, q)
            outs.append(_composite64(spec, net, o[r:q], d[r:q], t, dl, cnt, bounded))
    return {k: torch.cat([x[k] for x in outs]) for k in outs[0] if k != "eik" or kind == "render"}
