"""The serial tensor-core kernel where its rounds of tile pairs end (64-sample tiles: one per CTA,
pairs, a round and a rest of either kind) and the coarse-value kernel at the edges of its 256-sample
tiles.  A sample's result does not depend on the others in its launch, so the same ray rendered alone
and in a batch of any size has the same bits: no tolerance."""
import numpy as np
import pytest
import torch

from paper_2311_17878_gb300 import build, synth
from paper_2311_17878_gb300 import tsdfs as T

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    T.lib()


def render(mlp, n_rays, per_ray, o, d):
    b = T.Bounds(n_rays)
    b.t_n.fill_(0.5)
    b.t_f.fill_(2.5)
    b.status.fill_(T.TSDFS_BOUNDED)
    b.offsets.copy_(torch.arange(n_rays + 1, dtype=torch.int32) * per_ray)
    out = T.Renderer(mlp, n_rays, n_rays * per_ray).render(o[:n_rays].contiguous(), d[:n_rays].contiguous(), b)
    return torch.cat([out.rgb, out.depth[:, None], out.wsum[:, None], out.normal, out.eik[:, None]], 1)


@pytest.mark.parametrize("scene,precision", [("room", T.TSDFS_PREC_F16), ("tiny", T.TSDFS_PREC_BF16)])
def test_rest_tiles(scene, precision):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    o, d = (torch.tensor(a).cuda() for a in synth.room_heldout_rays(0))
    idx = torch.tensor(synth.sub_sample(len(o), 6 * sms, seed=3)).cuda()
    o, d = o[idx].contiguous(), d[idx].contiguous()
    mlp = T.Mlp(synth.scene_mlp(scene), precision)
    whole = render(mlp, 6 * sms, 64, o, d)      # one tile per ray, three rounds of pairs
    # tiles: 1, one per CTA, one more, a round of pairs, a round and singles, and pairs again
    for n in (1, sms, sms + 1, 2 * sms - 1, 2 * sms, 2 * sms + 3, 3 * sms, 3 * sms + 1, 5 * sms):
        assert torch.equal(render(mlp, n, 64, o, d), whole[:n]), n
    # samples that end inside a tile
    few = render(mlp, 5, 13, o, d)
    assert torch.equal(render(mlp, 100, 13, o, d)[:5], few)
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits


@pytest.mark.parametrize("scene,precision", [("room", T.TSDFS_PREC_F16), ("room", T.TSDFS_PREC_BF16), ("tiny", T.TSDFS_PREC_F16)])
def test_coarse_tiles(scene, precision):
    wl = synth.room_workload(with_views=False)
    g = T.Grid(wl.grid)
    o, d = (torch.tensor(a).cuda() for a in synth.room_heldout_rays(1))
    idx = torch.tensor(synth.sub_sample(len(o), 1500, seed=4)).cuda()
    o, d = o[idx].contiguous(), d[idx].contiguous()
    mlp = T.Mlp(synth.scene_mlp(scene), precision)

    def run(n):
        out = T.HierRenderer(mlp, n, n_coarse=64, n_fine=8).render(g, o[:n].contiguous(), d[:n].contiguous(), 0.05, 12.0)
        return torch.cat([out.rgb, out.depth[:, None], out.wsum[:, None], out.normal], 1)

    whole = run(1500)
    for n in (1, 2, 3, 4, 5, 609, 1499):
        assert torch.equal(run(n), whole[:n]), n
    assert np.isfinite(whole.cpu().numpy()).all()
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits


@pytest.mark.parametrize("scene,precision", [("room", T.TSDFS_PREC_BF16X2), ("tiny", T.TSDFS_PREC_BF16X2),
                                             ("room", T.TSDFS_PREC_F16)])
def test_pipelined_colour_layers_over_several_tiles(scene, precision):
    """The pipelined kernel runs the colour layers for up to four 32-sample tiles of a CTA at a time
    (here two tiles per ray): the bits of the rays in parts of one tile to a CTA."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    o, d = (torch.tensor(a).cuda() for a in synth.room_heldout_rays(0))
    half = sms // 2
    idx = torch.tensor(synth.sub_sample(len(o), 7 * half, seed=4)).cuda()
    o, d = o[idx].contiguous(), d[idx].contiguous()
    mlp = T.Mlp(synth.scene_mlp(scene), precision)
    before = T.tsdfs_network_kernel(precision)
    T.tsdfs_set_network_kernel(precision, T.TSDFS_NETKERNEL_PIPELINED)
    try:
        parts = torch.cat([render(mlp, half, 64, o[r:], d[r:]) for r in range(0, 7 * half, half)])
        # tiles per CTA: 1 and 2, 2, 4, 4 and 5, 5, 6, 7
        for n in (half + 1, 2 * half, 4 * half, 4 * half + 1, 5 * half, 6 * half, 7 * half):
            assert torch.equal(render(mlp, n, 64, o, d), parts[:n]), n
    finally:
        T.tsdfs_set_network_kernel(precision, before)
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits
