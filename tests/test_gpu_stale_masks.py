"""Blended-pair masks that an earlier forward left in the workspace must not
show.  The first forward blends every surfel at every pixel of the one tile; in
the second one a stack in front stops the tile's lower four rows early, while
the upper four go on.  Pair counts, attributed errors and gradients of the
second must be those of a workspace that never held the first."""
import pytest
import torch

from paper_2604_03092_gb300 import scenes
from paper_2604_03092_gb300.rasterizer import RasterConfig, Rasterizer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk,bwd_chunk", [(64, 64), (128, 64), (64, 256), (256, 128)])
def test_second_forward_sees_no_old_masks(chunk, bwd_chunk):
    front, n = 100, 450
    views = scenes.random_scene(n=1, width=8, height=8, f=8.0).views
    quats = torch.tensor([[1.0, 0.0, 0.0, 0.0]]).repeat(n, 1)
    means = torch.zeros(n, 3)
    means[:, 2] = torch.linspace(2.0, 3.0, n)
    scales, rgb = torch.full((n, 2), 8.0), torch.rand(n, 3, generator=torch.Generator().manual_seed(0))
    opacity = torch.full((n,), 0.015)
    first = [t.cuda() for t in (means, scales, quats, opacity, rgb)]
    # the stack: centred on the last rows, 1.2 pixels wide in y, opaque; the rest a little denser than before
    means, scales, opacity = means.clone(), scales.clone(), torch.full((n,), 0.03)
    means[:front, 1] = (7.0 - 4.0) / 8.0 * means[:front, 2]
    scales[:front, 1] = 1.2 / 8.0 * means[:front, 2]
    opacity[:front] = 0.99
    second = [t.cuda() for t in (means, scales, quats, opacity, rgb)]
    gen = torch.Generator().manual_seed(1)
    cfg = RasterConfig(chunk=chunk, bwd_chunk=bwd_chunk)

    def render(rast, prm):
        im = rast.forward(*prm)
        err = torch.rand(64, generator=gen.manual_seed(2)).cuda() + 0.5
        up = [torch.rand(t.numel(), generator=gen.manual_seed(3)).cuda() for t in (im.rgb, im.depth, im.normal, im.alpha)]
        worst = rast.max_error(err)
        return worst, rast.backward(*prm, up), rast.stats()

    used = Rasterizer(views, n, cfg)
    assert render(used, first)[2]["fwd_pairs_blended"] == 64 * n
    worst, grads, stats = render(used, second)
    want_worst, want, want_stats = render(Rasterizer(views, n, cfg), second)
    alpha = used.forward(*second).alpha.reshape(8, 8)
    assert (alpha[4:] > 0.999).all() and want_stats["fwd_pairs_blended"] < 64 * n  # rows stopped
    assert stats["fwd_pairs_blended"] == want_stats["fwd_pairs_blended"]
    assert stats["bwd_pairs_blended"] == stats["fwd_pairs_blended"]
    assert torch.equal(worst, want_worst)
    for a, b in zip(grads, want):  # sums of atomics in any order
        assert float((a - b).norm()) <= 1e-4 * float(b.norm())
