"""The render workspaces: what they are sized for by precision and architecture, and that the calls take any
workspace with the serial kernel's 10 MB of scratch, with the same results."""
import numpy as np
import pytest
import torch

from paper_2311_17878_gb300 import build, synth
from paper_2311_17878_gb300 import tsdfs as T

LEAST = 256 * 4 * 2 * (4096 + 768)   # bytes of scratch every render needs
PRECISIONS = {"f32": T.TSDFS_PREC_F32, "bf16": T.TSDFS_PREC_BF16, "f16": T.TSDFS_PREC_F16, "bf16x2": T.TSDFS_PREC_BF16X2}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    T.lib()


def scratch(arch, precision):
    import ctypes as C
    m = T.tsdfs_mlp()
    m.arch, m.precision = arch, precision
    T.lib().tsdfs_render_workspace_size.restype = C.c_size_t
    return T.lib().tsdfs_render_workspace_size(C.byref(m), C.c_int64(1), C.c_int64(0)) - 256


def test_scratch_follows_precision_and_architecture():
    for p in PRECISIONS.values():
        assert scratch(0, p) == LEAST, p
    assert 30e6 < scratch(1, PRECISIONS["f32"]) < 34e6
    for p in ("bf16", "f16", "bf16x2"):
        assert LEAST <= scratch(1, PRECISIONS[p]) < 16e6, p
    import ctypes as C
    assert T.lib().tsdfs_render_workspace_size(None, C.c_int64(1), C.c_int64(0)) - 256 == scratch(1, PRECISIONS["f32"])


def align(n):
    return (n + 255) // 256 * 256


@pytest.mark.gpu
@pytest.mark.parametrize("scene", ["tiny", "room"])
@pytest.mark.parametrize("precision", list(PRECISIONS))
@pytest.mark.parametrize("call", ["render", "hier", "hier_bounded"])
def test_least_workspace_gives_the_same_results(scene, precision, call):
    from test_gpu_f32_split import rays
    from test_gpu_hier_bounded import bounds_on_device
    from test_gpu_render import dev
    counts = [64, 3, 40, 64, 17] * 100          # more tiles than the fewest CTAs
    o, d, b = rays(scene, counts, seed=101)
    wl = synth.tiny_workload() if scene == "tiny" else synth.room_workload(with_views=False)
    n, total = len(o), sum(counts)
    mlp, least = T.Mlp(synth.scene_mlp(scene), PRECISIONS[precision]), T.Mlp(synth.scene_mlp("tiny"), T.TSDFS_PREC_F16)
    bb, o, d = bounds_on_device(b), dev(o), dev(d)
    g, bp = T.Grid(wl.grid), wl.bounds
    if call == "render":
        full, size = T.tsdfs_render_workspace_size(mlp, n, total), align(48 * total) + align(4 * total) + LEAST + 256
    elif call == "hier":
        full, size = T.tsdfs_hier_workspace_size(mlp, n), T.tsdfs_hier_workspace_size(least, n)
    else:
        full, size = T.tsdfs_hier_bounded_workspace_size(mlp, n, 8, total), T.tsdfs_hier_bounded_workspace_size(least, n, 8, total)

    def run(ws):
        out = T.RenderOut(n)
        for t in (out.rgb, out.depth, out.wsum, out.normal, out.eik):
            t.zero_()
        if call == "render":
            T.render_rays(mlp, o, d, bb.t_n, bb.t_f, bb.offsets, bb.status, total, out.rgb, out.depth, out.wsum, out.normal,
                          out.eik, ws)
        elif call == "hier":
            T.render_rays_hier(mlp, g, o, d, 33, 17, bp.t_near, bp.t_far, out.rgb, out.depth, out.wsum, out.normal, ws)
        else:
            T.render_rays_hier_bounded(mlp, o, d, bb.t_n, bb.t_f, bb.offsets, bb.status, 8, total, out.rgb, out.depth,
                                       out.wsum, out.normal, ws)
        rc, bits = T.tsdfs_sync_status()
        assert rc == 0, bits
        return [t.cpu().numpy() for t in (out.rgb, out.depth, out.wsum, out.normal, out.eik)]

    assert LEAST < size <= full
    old = T.tsdfs_network_kernel(PRECISIONS[precision]) if precision in ("f16", "bf16") else None
    kernels = [T.TSDFS_NETKERNEL_SERIAL, T.TSDFS_NETKERNEL_PIPELINED] if old else [None]
    try:
        for kernel in kernels:
            if kernel:
                T.tsdfs_set_network_kernel(PRECISIONS[precision], kernel)
            for a, r in zip(run(torch.empty(size, dtype=torch.uint8, device="cuda")),
                            run(torch.empty(full, dtype=torch.uint8, device="cuda"))):
                assert a.tobytes() == r.tobytes()
    finally:
        if old:
            T.tsdfs_set_network_kernel(PRECISIONS[precision], old)
    with pytest.raises(T.TsdfsError):
        run(torch.empty(size - 1, dtype=torch.uint8, device="cuda"))
    assert np.isfinite(run(torch.empty(full, dtype=torch.uint8, device="cuda"))[0]).all()
