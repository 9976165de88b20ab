"""Compositing with a warp per ray (few rays) against a thread per ray (many): the sums run in the
samples' order either way, so the same ray has the same bits in a batch on either side of the rule."""
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


@pytest.mark.parametrize("opacity", [T.TSDFS_OPACITY_NEUS, T.TSDFS_OPACITY_VOLSDF])
@pytest.mark.parametrize("precision", [T.TSDFS_PREC_F16, T.TSDFS_PREC_BF16X2])
def test_same_bits_on_either_side_of_the_rule(precision, opacity):
    n = 9000
    rng = np.random.default_rng(65)
    wl = synth.tiny_workload()
    idx = rng.choice(len(wl.rays_o), n)
    o, d = (torch.tensor(a[idx]).cuda() for a in (wl.rays_o, wl.rays_d))
    counts = rng.choice([0, 1, 2, 31, 32, 33, 64, 65, 97], n, p=[.1, .2, .3, .1, .1, .1, .05, .03, .02])
    status = rng.choice([T.TSDFS_BOUNDED, T.TSDFS_FALLBACK, T.TSDFS_MISS], n, p=[.8, .1, .1]).astype(np.uint8)
    spec = synth.scene_mlp("tiny")
    spec.opacity = opacity
    mlp = T.Mlp(spec, precision)

    def render(q):
        m = len(counts[q])
        b = T.Bounds(m)
        b.t_n.fill_(1.0)
        b.t_f.fill_(2.9)
        b.status.copy_(torch.tensor(status[q]))
        b.offsets.copy_(torch.tensor(np.concatenate([[0], np.cumsum(counts[q])]), dtype=torch.int32))
        out = T.Renderer(mlp, m, int(counts[q].sum())).render(o[q].contiguous(), d[q].contiguous(), b)
        return torch.cat([out.rgb, out.depth[:, None], out.wsum[:, None], out.normal, out.eik[:, None]], 1)

    whole = render(slice(0, n))
    for q in (slice(0, 1), slice(5, 600), slice(600, 8792)):
        assert torch.equal(render(q), whole[q]), q
    rc, bits = T.tsdfs_sync_status()
    assert rc == 0, bits
