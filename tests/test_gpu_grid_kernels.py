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
