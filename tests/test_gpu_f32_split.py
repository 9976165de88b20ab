"""The single-precision networks on split FP16 operands (mlp_f32.cu) against the FP64 oracle:
sample totals around the 32-sample tiles (128 in the samplers' coarse pass), and networks whose
operands leave the range of the parts, whose tiles the SIMT kernel evaluates again.  The bars are
those of the FP32 render (depth 1e-4 relative, colour 2e-3): the split keeps FP32 accuracy, and
beyond its range the SIMT kernel has it."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import cgrid
from oracle import render as orr
from paper_2311_17878_gb300 import build, synth
from paper_2311_17878_gb300 import tsdfs as T
from test_gpu_render import DEPTH_REL_F32, RGB_ABS, compare, dev, gpu_render, oracle_render

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    T.lib()


def rays(scene, counts, seed):
    """Rays through the scene with the given sample counts around its surface."""
    wl = synth.tiny_workload() if scene == "tiny" else synth.room_workload(with_views=False)
    rng = np.random.default_rng(seed)
    n = len(counts)
    if scene == "tiny":
        o, d = wl.rays_o, wl.rays_d
        t = wl.scene.ray_range(o.astype(np.float64), d.astype(np.float64))
        idx = rng.choice(np.nonzero(np.isfinite(t))[0], n)
    else:
        o, d = synth.room_heldout_rays(0)
        idx = rng.choice(len(o), n)
        t = np.full(len(o), np.nan)
        t[idx] = wl.scene.ray_range(o[idx].astype(np.float64), d[idx].astype(np.float64))
    o, d, t = o[idx], d[idx], t[idx]
    return o, d, dict(t_n=(t - 0.12).astype(np.float32), t_f=(t + 0.06).astype(np.float32),
                      n=np.asarray(counts, np.int32), status=np.ones(n, np.uint8))


def spec_of(scene):
    return synth.scene_mlp(scene)


@pytest.mark.parametrize("scene", ["tiny", "room"])
@pytest.mark.parametrize("counts", [[1], [31], [32], [33], [16, 0, 49], [20] * 37, [64] * 160 + [7]],
                         ids=["1", "31", "32", "33", "gap", "740", "10247"])
def test_totals_around_tiles(scene, counts):
    o, d, b = rays(scene, counts, seed=61)
    spec = spec_of(scene)
    got = gpu_render(spec, o, d, b)
    ref, raw = oracle_render(spec, o, d, b)
    compare(got, ref, depth_rel=DEPTH_REL_F32)
    eik = np.zeros(len(counts))
    np.add.at(eik, np.repeat(np.arange(len(counts)), counts), raw["eik"].detach().numpy())
    assert np.allclose(got["eik"], eik, rtol=1e-3, atol=1e-5)
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits


def scaled(spec, which, layer, factor, undo):
    """The spec with one layer's outputs scaled up and, where ``undo``, the next layer's inputs
    scaled back: the network stays near itself while the activations between leave the range."""
    layers = [(W.copy(), b.copy()) for W, b in getattr(spec, which)]
    W, b = layers[layer]
    layers[layer] = (W * np.float32(factor), b * np.float32(factor))
    if undo:
        W, b = layers[layer + 1]
        layers[layer + 1] = (W / np.float32(factor), b)
    return dataclasses.replace(spec, **{which: layers})


@pytest.mark.parametrize("scene", ["tiny", "room"])
@pytest.mark.parametrize("case", ["sdf hidden", "colour hidden", "weights", "gradient", "gradient, opaque"])
def test_out_of_range_tiles(scene, case):
    o, d, b = rays(scene, [24] * 40, seed=62)
    spec = spec_of(scene)
    if case == "sdf hidden":       # activations near 1e4 between layers 1 and 2
        spec = scaled(spec, "sdf", 1, 4e4, True)
    elif case == "colour hidden":  # ReLU is homogeneous: the same function
        spec = scaled(spec, "rgb", 1, 4e5, True)
    elif case == "weights":        # weights beyond the parts' range; the small inputs keep z in it
        spec = scaled(spec, "rgb", 0, 1e6, True)
    else:                          # |grad f| near 1e-6: below what the parts' floor leaves exact
        W, bb = spec.sdf[-1]
        W, bb = W.copy(), bb.copy()
        W[0] *= np.float32(1e-6)
        bb[0] *= np.float32(1e-6)
        sharp = 1e6 if case == "gradient, opaque" else 1.0   # with the opacity's scale undone, or nearly transparent
        spec = dataclasses.replace(spec, sdf=[*spec.sdf[:-1], (W, bb)], inv_s=spec.inv_s * sharp)
    got = gpu_render(spec, o, d, b)
    ref, _ = oracle_render(spec, o, d, b)
    if np.any(ref["wsum"] > 1e-3):
        compare(got, ref, depth_rel=DEPTH_REL_F32)
    else:
        assert np.max(np.abs(got["rgb"] - ref["rgb"])) < RGB_ABS and np.max(np.abs(got["wsum"] - ref["wsum"])) < RGB_ABS
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits


@pytest.mark.parametrize("scene,n_rays,big", [("tiny", 1, False), ("tiny", 131, False), ("room", 65, False),
                                              ("room", 40, True)])
def test_coarse_pass(scene, n_rays, big):
    """The value-only tiles (128 samples): 8 coarse values per ray, in and out of range."""
    o, d, _ = rays(scene, [1] * n_rays, seed=63)
    wl = synth.tiny_workload() if scene == "tiny" else synth.room_workload(with_views=False)
    spec = spec_of(scene)
    if big:
        spec = scaled(spec, "sdf", 1, 4e4, True)
    bp = wl.bounds
    t0, te, ok = cgrid.clip_rays(wl.grid, o, d, bp.t_near, bp.t_far, "f32")
    assert np.all(ok)
    g = T.Grid(wl.grid)
    out = T.HierRenderer(T.Mlp(spec), n_rays, n_coarse=8, n_fine=4).render(g, dev(o), dev(d), bp.t_near, bp.t_far)
    ref = orr.render_hier(orr.Net(spec), o, d, t0.astype(np.float64), te.astype(np.float64), 8, 4)
    got = {k: getattr(out, k).cpu().numpy() for k in ("rgb", "depth", "wsum", "normal")}
    compare(got, {k: ref[k].detach().numpy() for k in got}, depth_rel=DEPTH_REL_F32)
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits


@pytest.mark.parametrize("scene", ["tiny", "room"])
@pytest.mark.parametrize("counts,huge", [([64] * 304, False), ([64] * 304 + [33], False), ([50] * 250, True)],
                         ids=["full", "one-over", "marked"])
def test_colour_layers_over_several_tiles(scene, counts, huge):
    """Totals at which a CTA's colour layers take four tiles, four and one, and three with marks."""
    o, d, b = rays(scene, counts, seed=63)
    spec = spec_of(scene)
    if huge:
        spec = scaled(spec, "rgb", 1, 4e5, True)
    got = gpu_render(spec, o, d, b)
    ref, _ = oracle_render(spec, o, d, b)
    compare(got, ref, depth_rel=DEPTH_REL_F32)
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits


def test_rays_of_almost_no_weight():
    """Room rays whose samples lie in free space keep the SIMT kernel's bits: those of a network scaled by a
    power of two between two ReLU layers (the same FP32 function), all of whose tiles leave the parts' range."""
    counts = [1, 16, 17, 40] * 25
    o, d, b = rays("room", counts, seed=66)
    free = np.arange(len(counts)) % 8 >= 4
    b["t_f"] = np.where(free, b["t_n"] - 0.1, b["t_f"]).astype(np.float32)
    b["t_n"] = np.where(free, 0.4 * b["t_f"], b["t_n"]).astype(np.float32)
    spec = spec_of("room")
    got = gpu_render(spec, o, d, b)
    ref = gpu_render(scaled(spec, "rgb", 1, 2.0 ** 19, True), o, d, b)
    thin = ref["wsum"] < 9e-4
    assert 5 <= thin.sum() <= 60
    for k in ("rgb", "depth", "wsum", "normal"):
        assert np.array_equal(got[k][thin], ref[k][thin]), k
    compare(got, ref, depth_rel=DEPTH_REL_F32)
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits


@pytest.mark.parametrize("n_coarse", [8, 31, 32, 64])
def test_sampler_with_few_coarse_samples(n_coarse):
    """Room networks over the whole box: below 32 coarse samples the SIMT kernel's bits (those of a network
    scaled by a power of two between two ReLU layers, the same FP32 function), from there the split's."""
    o, d, _ = rays("room", [1] * 150, seed=67)
    wl = synth.room_workload(with_views=False)
    spec, bp = spec_of("room"), wl.bounds
    g = T.Grid(wl.grid)

    def render(spec):
        out = T.HierRenderer(T.Mlp(spec), len(o), n_coarse=n_coarse, n_fine=4).render(g, dev(o), dev(d), bp.t_near, bp.t_far)
        return {k: getattr(out, k).cpu().numpy() for k in ("rgb", "depth", "wsum", "normal")}

    got = render(spec)
    if n_coarse < 32:
        ref = render(scaled(spec, "rgb", 1, 2.0 ** 19, True))
        for k in got:
            assert np.array_equal(got[k], ref[k]), k
    else:
        t0, te, ok = cgrid.clip_rays(wl.grid, o, d, bp.t_near, bp.t_far, "f32")
        assert np.all(ok)
        ref = orr.render_hier(orr.Net(spec), o, d, t0.astype(np.float64), te.astype(np.float64), n_coarse, 4)
        compare(got, {k: ref[k].detach().numpy() for k in got}, depth_rel=DEPTH_REL_F32)
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits
