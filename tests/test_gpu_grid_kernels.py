"""The brick-culled fusion, the word-wise inside mask and the merged ray-casting fusion against the
oracle (or, for values the oracle has no case for, a plain PyTorch restatement): bit for bit, so
without tolerances, at sizes that are no multiples of a brick, a word or a pixel tile, with cameras
inside, outside, beside and turned away from the grid."""
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


def bits(a):
    a = np.ascontiguousarray(a)
    return a.view(np.uint32) if a.dtype == np.float32 else a.view(np.uint16)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def random_views(n, w, h, seed, spread):
    """Cameras anywhere within ``spread`` of the origin, looking anywhere (rolled too), some with
    mirrored or off-centre intrinsics; ranges of all sizes, some +inf."""
    rng = np.random.default_rng(seed)
    c2w, K = [], []
    for i in range(n):
        q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        c2w.append(np.concatenate([q, rng.uniform(-spread, spread, (3, 1))], 1).reshape(12))
        f = rng.uniform(0.3, 3.0) * w
        K.append([f * (-1 if i % 7 == 3 else 1), f * rng.uniform(0.7, 1.3), w * rng.uniform(-0.2, 1.2), h * rng.uniform(0, 1)])
    depth = rng.uniform(0.0, 2.5, (n, h, w)).astype(np.float32)
    depth[rng.random((n, h, w)) < 0.1] = np.inf
    return synth.Views(np.asarray(K, np.float32), np.asarray(c2w, np.float32), depth, w, h)


@pytest.mark.parametrize("shape,n_views,spread", [((32, 4, 4), 9, 1.5), ((1, 1, 1), 3, 0.5), ((70, 9, 13), 40, 1.0),
                                                  ((33, 37, 5), 300, 1.2), ((96, 40, 21), 25, 6.0)])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_culled_fusion_bit_exact(shape, n_views, spread, dtype):
    spec = synth.GridSpec(*shape, (-0.5, -0.4, -0.3), 1.0 / max(shape), 3.0 / max(shape), dtype)
    views = random_views(n_views, 23, 17, n_views, spread)
    g = T.Grid(spec).init().integrate(dev(views.depth), dev(views.K), dev(views.c2w))
    V, W = cgrid.integrate_projective(spec, views, "f32")
    assert np.array_equal(g.W.cpu().numpy(), W)
    got = g.V.cpu().numpy()
    assert np.array_equal(bits(got), bits(V) if V.dtype != np.uint16 else V)
    if n_views >= 25:
        assert W.max() > 0


def mask_ref(V, r):
    """-1 outside; a maximum that ignores NaN (torch's fmax) per axis, then < 0."""
    p = torch.nn.functional.pad(V, (r,) * 6, value=-1.0)
    for axis in range(3):
        n = V.shape[axis]
        m = p.narrow(axis, 0, n)
        for d in range(1, 2 * r + 1):
            m = torch.fmax(m, p.narrow(axis, d, n))
        p = m
    return p < 0


@pytest.mark.parametrize("shape", [(8, 8, 256), (9, 17, 288), (5, 3, 31), (11, 8, 33), (16, 9, 300), (1, 1, 1), (3, 2, 520)])
@pytest.mark.parametrize("r", [0, 1, 2, 4])
@pytest.mark.parametrize("nan", [False, True])
def test_mask_words(shape, r, nan):
    gen = torch.Generator().manual_seed(r + 10 * shape[2])
    V = torch.rand(shape, generator=gen) * 2 - 1.02
    # mostly negative, so that neighbourhoods pass
    V = torch.where(torch.rand(shape, generator=gen) < 0.02, V.abs(), -V.abs())
    V[torch.rand(shape, generator=gen) < 0.01] = -0.0
    if nan:
        V[torch.rand(shape, generator=gen) < 0.01] = float("nan")
        V[:2 * r + 1, :2 * r + 1, -40:] = float("nan")   # whole neighbourhoods of NaN
    nz, ny, nx = shape
    g = T.Grid(synth.GridSpec(nx, ny, nz, (0, 0, 0), 0.1, 0.3), V=V.cuda(), W=torch.zeros(shape, dtype=torch.uint8).cuda())
    words = g.inside_mask(r).cpu().numpy().view(np.uint32)
    got = np.unpackbits(words.view(np.uint8), bitorder="little")
    ref = mask_ref(V, r).numpy().reshape(-1)
    assert np.array_equal(got[:ref.size].astype(bool), ref)
    assert not got[ref.size:].any()


@pytest.mark.parametrize("shape,w,h", [((25, 25, 25), 8, 4), ((13, 21, 9), 41, 19), ((1, 1, 1), 3, 3), ((64, 31, 17), 130, 33)])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_merged_raycast_bit_exact(shape, w, h, dtype):
    spec = synth.GridSpec(*shape, (-0.5, -0.4, -0.3), 1.0 / max(shape), 3.0 / max(shape), dtype)
    views = random_views(6, w, h, w, 0.7)
    g = T.Grid(spec).init().integrate_raycast(dev(views.depth), dev(views.K), dev(views.c2w))
    V, W = cgrid.integrate_raycast_batched(spec, views, "f32")
    assert np.array_equal(g.W.cpu().numpy(), W)
    got = g.V.cpu().numpy()
    assert np.array_equal(bits(got), bits(V) if V.dtype != np.uint16 else V)


@pytest.mark.parametrize("n", [1, 31, 8191, 8192, 8193, 40000, 8192 * 70 + 5])
def test_scan_sizes(n):
    """Offsets of the adaptive counts: one chunk, its edges, several chunks."""
    rng = np.random.default_rng(n)
    b = T.Bounds(n)
    status = rng.choice([0, 1, 2], n).astype(np.uint8)
    b.t_n.copy_(dev(rng.uniform(0, 1, n).astype(np.float32)))
    b.t_f.copy_(b.t_n + dev(rng.uniform(0, 1, n).astype(np.float32)))
    b.status.copy_(dev(status))
    out = T.AdaptiveCounts(n).apply(b, n_mean=8, n_min=2, n_max=64, n_fallback=64)
    cnt = out.n.cpu().numpy().astype(np.int64)
    assert np.array_equal(out.offsets.cpu().numpy(), np.concatenate([[0], np.cumsum(cnt)]))


@pytest.mark.parametrize("n_rays", [1, 33, 500, 3000])
@pytest.mark.parametrize("radius,dtype", [(0, "f32"), (1, "f16"), (2, "f32"), (3, "f32"), (4, "f16")])
def test_few_rays_without_mask(n_rays, radius, dtype):
    """Far phase from the neighbourhoods themselves, at ray counts around its launch rule."""
    wl = synth.tiny_workload()
    spec = synth.GridSpec(**{**wl.grid.__dict__, "dtype": dtype})
    V, _ = cgrid.integrate_projective(spec, wl.views, "f32")
    rng = np.random.default_rng(n_rays)
    idx = rng.choice(len(wl.rays_o), n_rays)
    o, d = wl.rays_o[idx], wl.rays_d[idx]
    bp = synth.BoundsParams(**{**wl.bounds.__dict__, "nb_radius": radius, "m_confirm": 3})
    Vd = torch.as_tensor(V.view(np.float16) if dtype == "f16" else V).cuda()
    g = T.Grid(spec, V=Vd, W=torch.zeros(spec.shape_zyx, dtype=torch.uint8).cuda())
    got = T.Bounds(n_rays).compute(g, dev(o), dev(d), bp, None)
    ref = cgrid.ray_bounds(spec, V, o, d, bp, "f32")
    for k in ("n", "status"):
        assert np.array_equal(getattr(got, k).cpu().numpy(), ref[k]), k
    for k in ("t_n", "t_f"):
        assert np.array_equal(bits(getattr(got, k).cpu().numpy()), bits(ref[k].astype(np.float32))), k
    z, rz = got.t_zero.cpu().numpy(), ref["t_zero"].astype(np.float32)
    assert np.array_equal(np.isnan(z), np.isnan(rz)) and np.array_equal(z[~np.isnan(z)], rz[~np.isnan(rz)])


def degenerate(rng, o, d):
    """Some rays along an axis or a plane, on voxel boundaries, from inside, with a tiny component."""
    o, d = o.copy(), d.copy()
    k = len(o) // 16
    for j in range(k):
        kind = j % 6
        a = int(rng.integers(3))
        if kind == 0:
            d[j] = 0
            d[j, a] = rng.choice([-1.0, 1.0])
        elif kind == 1:
            d[j, a] = 0
        elif kind == 2:
            o[j] = np.round(o[j] * 8) / 8
            d[j] = rng.choice([-1.0, 1.0], 3)
        elif kind == 3:
            o[j] = rng.uniform(-0.4, 0.4, 3)
        elif kind == 4:
            d[j, a] = 1e-38 * rng.choice([-1.0, 1.0])
        else:
            d[j, a] = 1e-42
    n = np.linalg.norm(d, axis=1, keepdims=True)
    return o.astype(np.float32), (d / n).astype(np.float32)


@pytest.mark.parametrize("shape,dtype,dense", [((64, 64, 64), "f32", 0.001), ((61, 35, 83), "f16", 0.01), ((7, 9, 5), "f32", 0.2),
                                               ((100, 8, 16), "f32", 0.0), ((33, 64, 40), "f32", 0.5)])
@pytest.mark.parametrize("use_mask", [False, True])
@pytest.mark.parametrize("zero", [True, False])
def test_warp_per_ray_matches_thread_per_ray(shape, dtype, dense, use_mask, zero):
    """20 011 rays in one call (a thread per ray) against the same rays in calls below the rule's
    counts (a warp per ray): bit for bit."""
    rng = np.random.default_rng(shape[0])
    nx, ny, nz = shape
    vs = 1.0 / max(shape)
    spec = synth.GridSpec(nx, ny, nz, (-0.5 * nx * vs, -0.5 * ny * vs, -0.5 * nz * vs), vs, 3 * vs, dtype)
    z, y, x = np.meshgrid(*[np.linspace(-1, 1, k) for k in (nz, ny, nx)], indexing="ij")
    V = np.clip(4 * (np.sqrt(x * x + y * y + z * z) - 0.5), -1, 1).astype(np.float32)   # a ball
    spots = rng.random(V.shape) < dense
    V[spots] = rng.uniform(-1, 1, int(spots.sum()))
    n = 20011
    o = rng.normal(size=(n, 3))
    o /= np.linalg.norm(o, axis=1, keepdims=True)
    d = rng.uniform(-0.45, 0.45, (n, 3)) - o
    o, d = degenerate(rng, o, d / np.linalg.norm(d, axis=1, keepdims=True))
    bp = synth.BoundsParams(d_s=vs, t_near=0.0, t_far=4.0, step=vs, nb_radius=1, m_confirm=4, n_max=32)
    g = T.Grid(spec, V=torch.as_tensor(V).to(torch.float16 if dtype == "f16" else torch.float32).cuda(),
               W=torch.zeros(V.shape, dtype=torch.uint8).cuda())
    mask = g.inside_mask(1) if use_mask else None

    def compute(lo, hi):
        b = T.Bounds(hi - lo)
        T.tsdf_ray_bounds(g, mask, dev(o[lo:hi]), dev(d[lo:hi]), T.bounds_params(bp), b.t_n, b.t_f, b.n, b.offsets,
                          b.t_zero if zero else None, b.status, b.workspace)
        return {k: getattr(b, k).cpu().numpy() for k in ("t_n", "t_f", "n", "status") + (("t_zero",) if zero else ())}

    whole = compute(0, n)
    parts = [compute(a, min(n, a + 5000)) for a in range(0, n, 5000)]
    for k in whole:
        part = np.concatenate([q[k] for q in parts])
        assert np.array_equal(whole[k].view(np.uint8) if k == "status" else whole[k].view(np.uint32),
                              part.view(np.uint8) if k == "status" else part.view(np.uint32)), k
    assert (whole["status"] == 1).sum() > 1000 or dense == 0.0
