"""Fusion, inside mask and ray-casting fusion of small, thin and long grids, with few and many views, against the
oracle (the mask: a PyTorch restatement) bit for bit: the sizes at which their kernels change over."""
import numpy as np
import pytest
import torch

from oracle import cgrid
from paper_2311_17878_gb300 import build, synth
from paper_2311_17878_gb300 import tsdfs as T
from test_gpu_grid_kernels import bits, dev, mask_ref, random_views

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    T.lib()


@pytest.mark.parametrize("shape,n_views", [((1, 40, 37), 30), ((37, 1, 40), 30), ((40, 37, 1), 30), ((2, 300, 3), 90), ((1, 1, 700), 90),
                                           ((16, 16, 16), 60), ((64, 64, 64), 4), ((65, 64, 64), 4), ((8, 9, 8), 256), ((24, 20, 16), 257),
                                           ((24, 20, 16), 641), ((70, 66, 68), 640), ((70, 66, 68), 641), ((7, 200, 211), 3)])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_fusion(shape, n_views, dtype):
    spec = synth.GridSpec(*shape, (-0.5, -0.4, -0.3), 1.0 / max(shape), 3.0 / max(shape), dtype)
    views = random_views(n_views, 13, 11, n_views + shape[0], 1.1)
    g = T.Grid(spec).init().integrate(dev(views.depth), dev(views.K), dev(views.c2w))
    V, W = cgrid.integrate_projective(spec, views, "f32")
    assert np.array_equal(g.W.cpu().numpy(), W)
    got = g.V.cpu().numpy()
    assert np.array_equal(bits(got), bits(V) if V.dtype != np.uint16 else V)
    assert n_views < 9 or W.max() > 0


@pytest.mark.parametrize("shape", [(4, 4, 700), (90, 4, 40), (121, 96, 130), (128, 128, 128), (130, 128, 127), (1, 65, 513), (2000, 3, 5)])
@pytest.mark.parametrize("r", [0, 2, 4])
def test_mask(shape, r):
    gen = torch.Generator().manual_seed(r + shape[2])
    V = -torch.rand(shape, generator=gen)
    V = torch.where(torch.rand(shape, generator=gen) < 0.01, -V, V)
    V[torch.rand(shape, generator=gen) < 0.002] = float("nan")
    nz, ny, nx = shape
    g = T.Grid(synth.GridSpec(nx, ny, nz, (0, 0, 0), 0.1, 0.3), V=V.cuda(), W=torch.zeros(shape, dtype=torch.uint8).cuda())
    words = g.inside_mask(r).cpu().numpy().view(np.uint32)
    got = np.unpackbits(words.view(np.uint8), bitorder="little")
    ref = mask_ref(V, r).numpy().reshape(-1)
    assert np.array_equal(got[:ref.size].astype(bool), ref)
    assert not got[ref.size:].any()


@pytest.mark.parametrize("ny,nz", [(262141, 1), (1, 262141)])
def test_mask_refuses_what_it_refused(ny, nz):
    """More than 262 140 rows along an axis."""
    spec = synth.GridSpec(1, ny, nz, (0, 0, 0), 0.1, 0.3)
    g = T.Grid(spec).init()
    with pytest.raises(T.TsdfsError):
        g.inside_mask(1)


@pytest.mark.parametrize("shape,w,h,spread", [((20, 21, 22), 9, 7, 3.0), ((20, 21, 22), 1, 70, 0.4), ((64, 64, 64), 100, 3, 2.0),
                                              ((70, 69, 68), 90, 70, 0.9), ((90, 30, 100), 200, 150, 2.5), ((70, 70, 70), 33, 4, 0.3)])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_raycast(shape, w, h, spread, dtype):
    """Cameras in the grid, near it and far from it, whose pixels' rays share voxels or do not."""
    spec = synth.GridSpec(*shape, (-0.5, -0.4, -0.3), 1.0 / max(shape), 3.0 / max(shape), dtype)
    views = random_views(7, w, h, w + shape[1], spread)
    g = T.Grid(spec).init().integrate_raycast(dev(views.depth), dev(views.K), dev(views.c2w))
    V, W = cgrid.integrate_raycast_batched(spec, views, "f32")
    assert np.array_equal(g.W.cpu().numpy(), W)
    got = g.V.cpu().numpy()
    assert np.array_equal(bits(got), bits(V) if V.dtype != np.uint16 else V)
