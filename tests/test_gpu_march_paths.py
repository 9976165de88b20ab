"""The march's two kernels (a warp per ray, a thread per ray) beyond the sizes of the other tests: every launch
shape and the step cap on either side of the rule between them, and grids of 2^23 voxels on a side, which walk
in integers, against the oracle bit for bit."""
import numpy as np
import pytest
import torch

from oracle import cgrid
from paper_2311_17878_gb300 import build, synth
from paper_2311_17878_gb300 import tsdfs as T

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    T.lib()
    T.tsdfs_sync_status()


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


@pytest.fixture(scope="module")
def ball():
    """The sphere's volume, 20 011 rays on it, its inside mask and the oracle's bounds."""
    wl = synth.tiny_workload()
    V, _ = cgrid.integrate_projective(wl.grid, wl.views, "f32")
    idx = np.random.default_rng(81).choice(len(wl.rays_o), 20011)
    o, d = wl.rays_o[idx], wl.rays_d[idx]
    g = T.Grid(wl.grid, V=dev(V), W=torch.zeros(V.shape, dtype=torch.uint8, device="cuda"))
    return wl, g, o, d, g.inside_mask(wl.bounds.nb_radius), cgrid.ray_bounds(wl.grid, V, o, d, wl.bounds, "f32")


def compute(g, o, d, bp, mask):
    b = T.Bounds(len(o)).compute(g, dev(o), dev(d), bp, mask)
    return {k: getattr(b, k).cpu().numpy() for k in ("t_n", "t_f", "n", "status", "t_zero")}


def same(got, ref, n):
    for k in got:
        r = ref[k][:n].astype(got[k].dtype)
        assert np.array_equal(got[k], r, equal_nan=got[k].dtype.kind == "f"), k


# rays on either side of the rule, which is lower with the mask than without
SIDES = [(4096, True), (4097, True), (16384, False), (16385, False)]


@pytest.mark.parametrize("n,use_mask", SIDES)
@pytest.mark.parametrize("block,per_sm", [(32, 1), (64, 4), (128, 64), (256, 1), (256, 64)])
def test_launch_shapes(ball, n, use_mask, block, per_sm):
    wl, g, o, d, mask, ref = ball
    try:
        T.tsdfs_set_bounds_launch_shape(block, per_sm)
        same(compute(g, o[:n], d[:n], wl.bounds, mask if use_mask else None), ref, n)
    finally:
        T.tsdfs_set_bounds_launch_shape(0, 0)


def test_autotuned_shapes(ball):
    """The autotuner on few rays, then on many: its choice is what is read, and the outputs stay."""
    wl, g, o, d, mask, ref = ball
    try:
        for n in (3001, 20011):
            b = T.Bounds(n)
            block, per_sm, _ = b.autotune(g, dev(o[:n]), dev(d[:n]), wl.bounds, mask, reps=1)
            assert T.tsdfs_bounds_launch_shape() == (block, per_sm)
            for m in (3001, 20011):
                same(compute(g, o[:m], d[:m], wl.bounds, mask), ref, m)
    finally:
        T.tsdfs_set_bounds_launch_shape(0, 0)
    assert T.tsdfs_bounds_launch_shape() == (128, 64)


@pytest.mark.parametrize("n,use_mask", SIDES)
def test_step_cap(ball, n, use_mask):
    """A walk cut short after a few voxels reports it; the rays fall back to the whole clip, or keep t_f = t_end."""
    wl, g, o, d, mask, ref = ball
    t0, te, _ = cgrid.clip_rays(wl.grid, o[:n], d[:n], wl.bounds.t_near, wl.bounds.t_far, "f32")
    bounded = ref["status"][:n] == 1
    try:
        for cap in (4, 24):
            T.tsdfs_set_test_limits(0, cap, -1)
            got = compute(g, o[:n], d[:n], wl.bounds, mask if use_mask else None)
            rc, bits = T.tsdfs_sync_status()
            assert rc == T.TSDFS_E_DEVICE and bits & T.TSDFS_DEV_MARCH_CAP, bits
            cut, kept = bounded & (got["status"] == 2), bounded & (got["status"] == 1)
            assert np.array_equal(got["t_n"][cut], t0[cut]) and np.array_equal(got["t_f"][cut], te[cut])
            assert np.array_equal(got["t_n"][kept], ref["t_n"][:n][kept])
            short = kept & (got["t_f"] != ref["t_f"][:n])
            assert np.array_equal(got["t_f"][short], te[short])
            assert cut.sum() + short.sum() > 100
    finally:
        T.tsdfs_set_test_limits(0, 0, -1)
        T.tsdfs_sync_status()
    same(compute(g, o[:n], d[:n], wl.bounds, mask if use_mask else None), ref, n)


def long_grid(axis, dtype):
    """2^23 x 1 x 1 voxels of 2^-10 along an axis, from 0, with runs of either sign."""
    n = [1, 1, 1]
    n[axis] = 1 << 23
    spec = synth.GridSpec(*n, (0.0, 0.0, 0.0), 2.0 ** -10, 3 * 2.0 ** -10, dtype)
    i = np.arange(1 << 23)
    V = (np.where((i // 37) % 3 == 1, -1.0, 1.0) * (0.25 + (i * 2654435761 % 1024) / 1400.0)).astype(np.float32)
    V = V.reshape(n[2], n[1], n[0])
    return spec, V.astype(np.float16).view(np.uint16) if dtype == "f16" else V


@pytest.mark.parametrize("axis,dtype,use_mask", [(0, "f32", False), (0, "f16", True), (1, "f16", False), (2, "f32", False)])
@pytest.mark.parametrize("n", [257, 20011])
def test_long_grid(axis, dtype, use_mask, n):
    """Rays nearly along the axis, forwards and back, near the start, the middle and the end of the grid."""
    spec, V = long_grid(axis, dtype)
    rng = np.random.default_rng(82)
    side = np.float64(2.0 ** -10)
    o = rng.uniform(0.1, 0.9, (n, 3)) * side
    o[:, axis] = rng.choice([0.5, 100.0, 4096.0, 8191.0], n) + rng.uniform(-0.4, 0.4, n)
    d = rng.uniform(-1e-3, 1e-3, (n, 3))
    d[:, axis] = rng.choice([-1.0, 1.0], n)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    o, d = o.astype(np.float32), d.astype(np.float32)
    bp = synth.BoundsParams(d_s=float(side), t_near=0.0, t_far=0.5, step=float(2 * side), nb_radius=1, m_confirm=3, n_max=32)
    Vd = torch.as_tensor(V.view(np.float16) if dtype == "f16" else V).cuda()
    g = T.Grid(spec, V=Vd, W=torch.zeros(spec.shape_zyx, dtype=torch.uint8).cuda())
    got = compute(g, o, d, bp, g.inside_mask(1) if use_mask else None)
    ref = cgrid.ray_bounds(spec, V, o, d, bp, "f32")
    same(got, ref, n)
    assert (got["status"] == 1).sum() > n // 2
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits


@pytest.mark.parametrize("axis", [0, 2])
def test_long_grid_raycast_fusion(axis):
    """Pixels' rays along a grid of 2^23 voxels that end after some hundred of them."""
    spec, _ = long_grid(axis, "f32")
    rng = np.random.default_rng(83)
    side = 2.0 ** -10
    w, h, n = 9, 7, 3
    c2w = []
    for k in range(n):
        fwd = np.zeros(3)
        fwd[axis] = 1.0
        right = np.roll(fwd, 1)
        pos = 0.5 * side * np.ones(3)
        pos[axis] = [0.25, 4096.0, 8190.0][k]
        c2w.append(np.concatenate([np.stack([right, np.cross(fwd, right), fwd], 1), pos[:, None]], 1).reshape(12))
    K = np.tile(np.array([2000.0, 2000.0, 4.5, 3.5], np.float32), (n, 1))
    depth = rng.uniform(0.05, 0.3, (n, h, w)).astype(np.float32)
    views = synth.Views(K, np.asarray(c2w, np.float32), depth, w, h)
    g = T.Grid(spec).init().integrate_raycast(dev(depth), dev(K), dev(views.c2w))
    V, W = cgrid.integrate_raycast_batched(spec, views, "f32")
    assert W.max() > 0
    assert np.array_equal(g.W.cpu().numpy(), W)
    assert np.array_equal(g.V.cpu().numpy().view(np.uint32), V.view(np.uint32))
