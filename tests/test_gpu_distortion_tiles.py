"""The depth distortion through every form of the 8x8 forward: whole tiles
(more than 18 per SM) and halves, center and ray depth, tails handed over at
once, on the way and at the default, at each chunk size (the distortion and
the depth sum it needs go through the hand-over).  Map and gradients against
the FP64 oracle; the other outputs are those of a render without it."""
import numpy as np
import pytest
import torch

import oracle
from gpu_utils import GRAD_REL_L2, oracle_cfg, rel_l2, to_dev, upstream
from paper_2604_03092_gb300 import scenes
from paper_2604_03092_gb300.rasterizer import RasterConfig, Rasterizer

pytestmark = pytest.mark.gpu

DIST_ATOL = 2e-5  # FP32 accumulation of 2 w (z A - D) over up to ~150 blended pairs of depths up to 4 m


@pytest.mark.parametrize("ray", [False, True])
@pytest.mark.parametrize("n,width,height,f,chunk,tail", [
    (3000, 648, 520, 160.0, 128, 0),    # 5265 tiles: one warp per whole tile
    (3000, 648, 520, 160.0, 64, 20),
    (3000, 648, 520, 160.0, 64, 255),
    (1200, 40, 24, 32.0, 64, 255),
    (1200, 40, 24, 32.0, 64, 20),
    (1100, 40, 23, 32.0, 128, 255),
    (1100, 40, 23, 32.0, 128, 12),
    (900, 24, 20, 20.0, 256, 255),
    (1200, 40, 24, 32.0, 256, 0),
])
def test_distortion(n, width, height, f, chunk, tail, ray):
    sc = scenes.random_scene(n=n, width=width, height=height, f=f, seed=n + chunk, scale_range=(0.03, 0.2))
    sc.opacity = np.clip(sc.opacity * 0.5, 0.01, 0.99).astype(np.float32)
    cfg = RasterConfig(bg=(0.2, 0.1, 0.3), depth_ray=ray, chunk=chunk, fwd_tail=tail)
    params = to_dev(sc)
    plain = Rasterizer(sc.views, sc.n, cfg).forward(*params)
    rast = Rasterizer(sc.views, sc.n, cfg)
    dist = torch.full((rast.n_pixels,), 7.0, device="cuda")
    im = rast.forward(*params, dist=dist)
    for a, b in zip(im, plain):
        assert torch.equal(a, b)
    d_dev, d_views = upstream(rast, 3)
    gd = np.random.default_rng(4).normal(size=(height, width)) * 5.0
    grads = rast.backward(*params, d_dev, d_dist=torch.from_numpy(gd.reshape(-1).astype(np.float32)).cuda())
    torch.cuda.synchronize()
    p = oracle.preprocess_scene_view(sc, 0, oracle_cfg(cfg))
    ref, flags = oracle.render_dist(p), oracle.render(p).pflags
    ok = (flags & (oracle.PF_FORWARD | (oracle.PF_BRANCH if ray else 0))) == 0
    assert ok.mean() > 0.99 and ref.max() > 1e-2
    err = np.abs(dist.view(height, width).cpu().numpy().astype(np.float64) - ref)[ok]
    assert err.max() <= DIST_ATOL, err.max()
    og = oracle.render_bwd(sc.means, sc.scales, sc.quats, p, d_views[0], g_dist=gd)
    out = {k: rel_l2(getattr(grads, k).cpu().numpy(), getattr(og, k)) for k in ("means", "scales", "quats", "opacity", "rgb")}
    out["pose"] = rel_l2(grads.pose.cpu().numpy()[0], og.pose)
    assert max(out.values()) <= GRAD_REL_L2, out
