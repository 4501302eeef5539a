"""Several views, each with a range of surfels of its own (uneven ranges, one
of a single surfel, an empty one, surfels that no view has): records, images
and gradients are those of the general path, where every range has two
views."""
import numpy as np
import pytest
import torch

from gpu_utils import rel_l2
from paper_2604_03092_gb300 import scenes
from paper_2604_03092_gb300.rasterizer import RasterConfig, Rasterizer

pytestmark = pytest.mark.gpu

RANGES = [(0, 700), (700, 1), (701, 0), (705, 12000), (12705, 17000)]


@pytest.mark.parametrize("tile", [8, 16])
def test_groups_of_one_view_equal_general_path(tile):
    n, w, h = 30_000, 203, 149
    sc = scenes.random_scene(n=n, width=w, height=h, f=170.0, seed=5, depth_range=(-4.0, 12.0), xy_range=6.0,
                             scale_range=(0.01, 0.3), n_views=len(RANGES))
    sc.means[700] = (0.1, 0.1, 3.0)
    prm = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (sc.means, sc.scales, sc.quats, sc.opacity, sc.rgb)]
    views = [scenes.View(w, h, 170.0, 165.0, 90.0, 80.0, v.Rt, off, cnt) for v, (off, cnt) in zip(sc.views, RANGES)]
    cfg = RasterConfig(tile_w=tile, tile_h=tile)
    one = Rasterizer(views, n, cfg)
    two = Rasterizer([v for v in views for _ in range(2)], n, cfg)
    im1, im2 = one.forward(*prm), two.forward(*prm)
    nt1 = one.ws_tensor(one.layout.ntiles, one.n_records, torch.int32)
    nt2 = two.ws_tensor(two.layout.ntiles, two.n_records, torch.int32)
    rec1 = one.ws_tensor(one.layout.records, 20 * one.n_records, torch.int32).view(-1, 20)
    rec2 = two.ws_tensor(two.layout.records, 20 * two.n_records, torch.int32).view(-1, 20)
    at = 0
    for _, cnt in RANGES:
        a, b = slice(at, at + cnt), slice(2 * at, 2 * at + cnt)
        assert torch.equal(nt1[a], nt2[b])
        inside = nt1[a] != 0
        assert cnt < 2 or 0 < int(inside.sum()) < cnt
        assert torch.equal(rec1[a][inside], rec2[b][inside])
        at += cnt
    for v in range(len(RANGES)):
        for a, b in zip(one.view_images(im1, v), two.view_images(im2, 2 * v)):
            assert torch.equal(a, b)
    gen = torch.Generator(device="cuda").manual_seed(1)
    d = [torch.randn(len(RANGES), c, h * w, device="cuda", generator=gen) for c in (3, 1, 3, 1)]
    g1 = one.backward(*prm, [t.reshape(-1) for t in d])
    # the general path with the second view of each range at zero
    g2 = two.backward(*prm, [torch.stack([t, torch.zeros_like(t)], 1).reshape(-1) for t in d])
    st1, st2 = one.stats(), two.stats()
    assert st1["status"] == 0 and st2["status"] == 0 and 2 * st1["n_visible"] == st2["n_visible"]
    for a, b in zip(g1[:5], g2[:5]):  # sums that meet in atomics: as vectors, far below the parity bar of 1e-3
        assert rel_l2(a.cpu().numpy(), b.cpu().numpy()) < 1e-5
    assert rel_l2(g1.pose.cpu().numpy(), g2.pose.cpu().numpy()[::2]) < 1e-5
    covered = torch.zeros(n, dtype=torch.bool, device="cuda")
    for off, cnt in RANGES:
        covered[off:off + cnt] = True
    assert not any(bool(t[~covered].any()) for t in g1[:5])
