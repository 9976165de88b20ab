"""Compositing with a warp per ray at the sample counts where its prefix sums change length (2, 8) and
where a row of 32 ends, against a thread per ray: the same bits."""
import pytest
import torch

from paper_2311_17878_gb300 import build, synth
from paper_2311_17878_gb300 import tsdfs as T

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    T.lib()


@pytest.mark.parametrize("count", [1, 2, 3, 7, 8, 9, 31, 32, 33, 34, 35, 40, 41])
def test_same_bits_for_every_length(count):
    n, few = 8300, 700
    wl = synth.tiny_workload()
    idx = torch.arange(n) * 7 % len(wl.rays_o)
    o, d = (torch.as_tensor(a)[idx].cuda() for a in (wl.rays_o, wl.rays_d))
    mlp = T.Mlp(synth.scene_mlp("tiny"), T.TSDFS_PREC_F16)

    def render(m):
        b = T.Bounds(m)
        b.t_n.fill_(1.0)
        b.t_f.fill_(2.9)
        b.status.fill_(T.TSDFS_BOUNDED)
        b.offsets.copy_(torch.arange(m + 1, dtype=torch.int32) * count)
        out = T.Renderer(mlp, m, m * count).render(o[:m].contiguous(), d[:m].contiguous(), b)
        return torch.cat([out.rgb, out.depth[:, None], out.wsum[:, None], out.normal, out.eik[:, None]], 1)

    whole = render(n)       # above 8192 rays: a thread per ray
    assert bool(torch.isfinite(whole).all())
    assert float(whole[:few, 4].max()) > 1e-3
    assert torch.equal(render(few), whole[:few])
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits
