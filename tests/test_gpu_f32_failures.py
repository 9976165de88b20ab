"""The bounded waits of the split FP32 network kernel (mlp_f32.cu), made to run out by weight items that are never
copied: the status word tells, compositing writes zeros, and the next call on the same context is right."""
import numpy as np
import pytest
import torch

from oracle import cgrid
from oracle import render as orr
from paper_2311_17878_gb300 import build, synth
from paper_2311_17878_gb300 import tsdfs as T
from test_gpu_f32_split import rays, spec_of
from test_gpu_render import DEPTH_REL_F32, compare, dev, gpu_render, oracle_render

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    T.lib()
    T.tsdfs_sync_status()


@pytest.fixture
def limits():
    yield T.tsdfs_set_test_limits
    T.tsdfs_set_test_limits(0, 0, -1)
    T.tsdfs_sync_status()


# withheld items of the SDF layers, of the colour layers, and of a later tile
@pytest.mark.parametrize("scene,item", [("tiny", 0), ("tiny", 5), ("room", 1), ("room", 5), ("room", 60), ("room", 200)])
def test_network_wait_runs_out_and_context_recovers(limits, scene, item):
    counts = [64] * (500 if item == 200 else 40)
    o, d, b = rays(scene, counts, seed=91)
    spec = spec_of(scene)
    limits(1 << 14, 0, item)
    got = gpu_render(spec, o, d, b)
    rc, bits = T.tsdfs_sync_status()
    assert rc == T.TSDFS_E_DEVICE and bits & T.TSDFS_DEV_TIMEOUT, bits
    for k in ("rgb", "wsum", "depth", "normal", "eik"):
        assert np.all(got[k] == 0), k
    limits(0, 0, -1)
    got = gpu_render(spec, o[:40], d[:40], {k: v[:40] for k, v in b.items()})
    rc, bits = T.tsdfs_sync_status()
    assert rc == T.TSDFS_OK and bits == 0
    ref, _ = oracle_render(spec, o[:40], d[:40], {k: v[:40] for k, v in b.items()})
    compare(got, ref, depth_rel=DEPTH_REL_F32)


@pytest.mark.parametrize("scene,n_coarse", [("tiny", 8), ("room", 33)])
def test_coarse_pass_wait_runs_out_and_context_recovers(limits, scene, n_coarse):
    o, d, _ = rays(scene, [1] * 100, seed=92)
    wl = synth.tiny_workload() if scene == "tiny" else synth.room_workload(with_views=False)
    spec, bp = spec_of(scene), wl.bounds
    h, g = T.HierRenderer(T.Mlp(spec), len(o), n_coarse=n_coarse, n_fine=4), T.Grid(wl.grid)
    limits(1 << 14, 0, 1)
    h.render(g, dev(o), dev(d), bp.t_near, bp.t_far)
    rc, bits = T.tsdfs_sync_status()
    assert rc == T.TSDFS_E_DEVICE and bits & T.TSDFS_DEV_TIMEOUT, bits
    limits(0, 0, -1)
    out = h.render(g, dev(o), dev(d), bp.t_near, bp.t_far)
    rc, bits = T.tsdfs_sync_status()
    assert rc == T.TSDFS_OK and bits == 0
    t0, te, _ = cgrid.clip_rays(wl.grid, o, d, bp.t_near, bp.t_far, "f32")
    with torch.no_grad():
        ref = orr.render_hier(orr.Net(spec), o, d, t0.astype(np.float64), te.astype(np.float64), n_coarse, 4)
    got = {k: getattr(out, k).cpu().numpy() for k in ("rgb", "depth", "wsum", "normal")}
    compare(got, {k: ref[k].detach().numpy() for k in got}, depth_rel=DEPTH_REL_F32)


def test_no_rerun_of_thin_rays_after_a_timeout(limits):
    """All weights are 0 then, but no ray is thin: the SIMT kernel, which takes a millisecond per 16 samples of a
    CTA, is not asked for them again."""
    counts = [64] * 2000
    o, d, b = rays("room", counts, seed=93)
    spec = spec_of("room")
    mlp = T.Mlp(spec)
    r = T.Renderer(mlp, len(o), sum(counts))
    bb = T.Bounds(len(o))
    bb.t_n.copy_(dev(b["t_n"]))
    bb.t_f.copy_(dev(b["t_f"]))
    bb.status.copy_(dev(b["status"]))
    bb.offsets.copy_(dev(np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)))
    oo, dd = dev(o), dev(d)
    # for scale, SIMT over all samples: a network out of range everywhere
    big = T.Mlp(spec)
    big.sdf_w.mul_(1e5)
    rb = T.Renderer(big, len(o), sum(counts))

    def ms(renderer):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        renderer.render(oo, dd, bb)
        e0.record()
        renderer.render(oo, dd, bb)
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1)

    simt = ms(rb)
    limits(1 << 10, 0, 5)
    late = ms(r)
    rc, bits = T.tsdfs_sync_status()
    assert rc == T.TSDFS_E_DEVICE and bits & T.TSDFS_DEV_TIMEOUT, bits
    assert late < 0.5 * simt, (late, simt)
