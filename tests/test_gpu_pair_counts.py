"""fwd_pairs_evaluated counts a pixel's pairs up to the one that stops it,
whatever the kernel computes beyond: the warp-per-tile forward of 8x8 tiles
(half tiles, whole tiles, dense chunks, tails) counts what the forward of
16x16 tiles does, which walks each pixel's entries one by one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,width,height,views,scales,kw", [
    (4000, 128, 96, 2, (0.01, 0.1), {}),                      # few tiles
    (20000, 333, 251, 2, (0.01, 0.1), {}),                    # 2688 tiles, dense chunks
    (60000, 333, 251, 1, (0.005, 0.03), {"depth_ray": True}),
    (60000, 640, 520, 1, (0.005, 0.03), {}),                  # 5200 tiles, sparse chunks
    (30000, 640, 520, 1, (0.01, 0.1), {"depth_ray": True}),
    (20000, 333, 251, 2, (0.01, 0.1), {"fwd_tail": 255}),
    (20000, 333, 251, 2, (0.01, 0.1), {"fwd_tail": 1, "chunk": 64}),
])
@pytest.mark.parametrize("distortion", [False, True])
def test_pairs_up_to_the_stop(n, width, height, views, scales, kw, distortion):
    import torch
    from paper_2604_03092_gb300 import scenes
    from paper_2604_03092_gb300.rasterizer import RasterConfig, Rasterizer

    sc = scenes.random_scene(n=n, width=width, height=height, f=100.0 * width / 128, seed=11, n_views=views,
                             scale_range=scales)
    # opaque surfels: nearly every pixel stops
    params = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
              for a in (sc.means, sc.scales, sc.quats, 0.5 + 0.5 * sc.opacity, sc.rgb)]
    counts = {}
    for tile in (8, 16):
        rast = Rasterizer(sc.views, sc.n, RasterConfig(tile_w=tile, tile_h=tile, **kw))
        dist = torch.empty(rast.n_pixels, device="cuda") if distortion else None
        rast.forward(*params, dist=dist)
        st = rast.stats()
        counts[tile] = np.array([st["fwd_pairs_evaluated"], st["fwd_pairs_blended"]])
    # the two take a pixel's transmittance in products of different order in
    # their tails: a few ulp, which puts a stop (at steps of some 10% and more
    # of T) on its other side once in 1e5 pixels or less, and moves the counts
    # by the entries up to the next that would stop it
    assert np.all(np.abs(counts[8] - counts[16]) <= 16 + 1e-6 * counts[16]), counts
