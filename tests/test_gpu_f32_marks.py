"""The samples that the split FP32 networks (mlp_f32.cu) hand to the SIMT kernel: which samples those are
depends on the sample alone, so a ray has the same bits in every batch; the coarse pass's marked
values against the FP64 oracle, at totals around the halves of its 128-sample tiles; and networks whose
operands come near the floor of the parts."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import cgrid
from oracle import render as orr
from paper_2311_17878_gb300 import build, synth
from paper_2311_17878_gb300 import tsdfs as T
from test_gpu_f32_split import rays, scaled, spec_of
from test_gpu_hier_bounded import bounds_on_device, render_gpu
from test_gpu_render import DEPTH_REL_F32, compare, dev, gpu_render

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    T.lib()


def mixed_batch(scene, kind):
    """Ordinary rays among rays that are handed over: of almost no weight, or too far out for the parts."""
    counts = [1, 5, 16, 17, 40, 3] * 20
    o, d, b = rays(scene, counts, seed=71)
    odd = np.arange(len(counts)) % 7 == 2
    if kind == "thin":
        b["t_f"] = np.where(odd, b["t_n"] - 0.1, b["t_f"]).astype(np.float32)
        b["t_n"] = np.where(odd, 0.4 * b["t_f"], b["t_n"]).astype(np.float32)
    else:
        b["t_n"] = np.where(odd, b["t_n"] + 1e5, b["t_n"]).astype(np.float32)
        b["t_f"] = np.where(odd, b["t_n"] + 1.0, b["t_f"]).astype(np.float32)
    return o, d, b


@pytest.mark.parametrize("sampler", ["bounded", "coarse and fine"])
@pytest.mark.parametrize("scene,kind", [("room", "thin"), ("room", "far"), ("tiny", "far")])
def test_a_ray_has_the_same_bits_in_every_batch(scene, kind, sampler):
    o, d, b = mixed_batch(scene, kind)
    spec = spec_of(scene)

    def render(idx):
        part = {k: v[idx] for k, v in b.items()}
        if sampler == "bounded":
            return gpu_render(spec, o[idx], d[idx], part)
        return render_gpu(spec, o[idx], d[idx], bounds_on_device(part), 8)

    n = len(o)
    whole = render(np.arange(n))
    rng = np.random.default_rng(72)
    for parts in ([np.arange(i, n, 7) for i in range(7)], np.array_split(np.arange(n), 9), [rng.permutation(n)]):
        for idx in parts:
            got = render(idx)
            for k in got:
                assert got[k].tobytes() == whole[k][idx].tobytes(), k
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits


@pytest.mark.parametrize("scene,n_rays,n_coarse", [("tiny", 133, 8), ("tiny", 139, 8), ("tiny", 1, 2), ("room", 40, 33),
                                                   ("room", 42, 33), ("room", 41, 64)])
def test_marked_coarse_values(scene, n_rays, n_coarse):
    """Every coarse value out of the parts' range; totals 40, 88 and 2, 40, 106 and 64 past a tile."""
    o, d, _ = rays(scene, [1] * n_rays, seed=73)
    wl = synth.tiny_workload() if scene == "tiny" else synth.room_workload(with_views=False)
    spec, bp = scaled(spec_of(scene), "sdf", 1, 4e4, True), wl.bounds
    t0, te, ok = cgrid.clip_rays(wl.grid, o, d, bp.t_near, bp.t_far, "f32")
    assert np.all(ok)
    out = T.HierRenderer(T.Mlp(spec), n_rays, n_coarse=n_coarse, n_fine=4).render(T.Grid(wl.grid), dev(o), dev(d),
                                                                                 bp.t_near, bp.t_far)
    got = {k: getattr(out, k).cpu().numpy() for k in ("rgb", "depth", "wsum", "normal")}
    with torch.no_grad():
        ref = orr.render_hier(orr.Net(spec), o, d, t0.astype(np.float64), te.astype(np.float64), n_coarse, 4)
    compare(got, {k: ref[k].detach().numpy() for k in got}, depth_rel=DEPTH_REL_F32)
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits


def near_the_floor(spec, case):
    """The spec with operands of some layers so small that FP16 parts of a fixed scale have few bits left, and
    the scale given back in the output layer, which takes no parts."""
    nets = {"sdf": [(W.copy(), b.copy()) for W, b in spec.sdf], "rgb": [(W.copy(), b.copy()) for W, b in spec.rgb]}

    def mul(net, layer, w, b):
        W, bb = nets[net][layer]
        nets[net][layer] = (W * np.float32(w), bb * np.float32(b))

    n = len(nets["sdf"])
    if case == "weights":            # of the last hidden layer: 1e-9 to 1e-7
        mul("sdf", n - 2, 1e-7, 1e-7)
        back = 1e7
    elif case == "tangents":         # 2e-9 between two hidden layers whose weights are 1e-6 to 1e-4
        for layer in ((0, 1) if n == 4 else (n - 4, n - 3)):
            mul("sdf", layer, 1e-4, 1e-4)
        back = 1e8
    else:                            # colour activations of 1e-11; ReLU is homogeneous: the same function
        for layer, (w, b) in enumerate([(1e-3, 1e-3), (1e-4, 1e-7), (1e-4, 1e-11), (1.0, 1e-11), (1e11, 1.0)]):
            mul("rgb", layer, w, b)
        return dataclasses.replace(spec, rgb=nets["rgb"])
    W, b = nets["sdf"][-1]
    W[0] *= np.float32(back)
    return dataclasses.replace(spec, sdf=nets["sdf"])


@pytest.mark.parametrize("scene,case", [("tiny", "weights"), ("tiny", "tangents"), ("room", "weights"), ("room", "tangents"),
                                        ("room", "colours")])
def test_operands_near_the_floor(scene, case):
    """One sample to a ray, so that its normal and colour are the ray's; through the sampler without fine
    samples, which has no rule for thin rays.  Every sample is handed over: the SDF cases have the SIMT kernel's
    bits, those of a network scaled by a power of two between two ReLU layers (the same FP32 function), which is
    out of range everywhere; the parts alone are 3e-5 to 1e-3 away in the normals, 1e-2 in the colours."""
    o, d, b = rays(scene, [1] * 300, seed=74)
    b["t_f"] = (b["t_n"] + np.linspace(0.02, 0.3, 300)).astype(np.float32)
    spec = near_the_floor(spec_of(scene), case)
    got = render_gpu(spec, o, d, bounds_on_device(b), 0)
    if case == "colours":
        with torch.no_grad():
            ref = orr.render_hier_bounded(orr.Net(spec), o, d, b["t_n"].astype(np.float64), b["t_f"].astype(np.float64),
                                          b["n"], 0)
        ref = {k: ref[k].detach().numpy() for k in ("rgb", "wsum")}
        live = ref["wsum"] > 1e-2
        assert live.sum() > 20
        off = np.abs(got["rgb"] / got["wsum"][:, None] - ref["rgb"] / ref["wsum"][:, None])[live]
        assert off.max() < 2e-5
    else:
        ref = render_gpu(scaled(spec, "rgb", 1, 2.0 ** 19, True), o, d, bounds_on_device(b), 0)
        for k in got:
            assert got[k].tobytes() == ref[k].tobytes(), k
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits
